"""The device calls captured into a CUDA graph: every replay gives the bits of a plain call.

The kernels of a call depend on one another through programmatic launches, of which a graph keeps only the edges between
neighbours: a kernel that begins before its predecessor has ended must not end before it, or what follows reads results that are
not there yet.  The handle's kernels are chosen so that the small dilations, which go first, take many times as long as the large ones.
"""
import numpy as np
import pytest

import paper_2301_08527_b200 as rk
from rocket_inputs import ar1_spike_series, kernels_from_lists, normal_array

pytestmark = pytest.mark.gpu


def _handle(C, L, small, large):
    rng = np.random.default_rng(C + L)
    ks = []
    for i in range(small + large):
        ln = (7, 9, 11)[i % 3]
        d = 1 if i < small else 130 + i
        m = min(C, 4) if i < small else 1
        ks.append(dict(dilation=d, padding=(ln - 1) * d // 2 if i % 2 else 0, channels=sorted(rng.choice(C, m, replace=False).tolist()),
                       weights=rng.normal(size=(m, ln)), bias=float(rng.uniform(-1, 1))))
    return rk.RocketParams.from_kernel_params(kernels_from_lists(C, L, ks))


# 6,001 steps: the tile kernels; 2,001: the kernel that holds whole examples, which has no neighbour but in the backward
@pytest.mark.parametrize("L,small,large", [(6001, 400, 2), (6001, 3, 200), (6001, 50, 0), (2001, 40, 30)])
def test_captured_calls_give_the_bits_of_plain_calls(L, small, large):
    import torch
    C, N = 6, 5
    p = _handle(C, L, small, large)
    K = small + large
    X = torch.from_numpy(ar1_spike_series(3, N, C, L)).cuda()
    g = torch.from_numpy(normal_array(4, (N, 2 * K))).cuda()
    p.reserve(N, rk.PASS_HARD | rk.PASS_SOFT | rk.PASS_BACKWARD)

    def calls(out):
        rk.rocket_transform(p, X, out=out["hard"])
        rk.rocket_transform_f16(p, X, out=out["half"])
        rk.rocket_transform_soft(p, X, 10.0, 3.0, out=out["soft"], argmax_out=out["arg"])
        rk.rocket_transform_soft_backward(p, X, 10.0, 3.0, g, out["arg"], out["dW"], out["db"])

    def buffers():
        z = lambda *s, dtype=torch.float32: torch.full(s, -7, dtype=dtype, device="cuda")  # noqa: E731
        return {"hard": z(N, 2 * K), "half": z(N, 2 * K), "soft": z(N, 2 * K), "arg": z(N, K, dtype=torch.int32),
                "dW": z(p.n_weights), "db": z(K)}

    want, got = buffers(), buffers()
    calls(want)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls(got)
    for _ in range(5):
        for t in got.values():
            t.fill_(-7)
        graph.replay()
        torch.cuda.synchronize()
        for name, t in want.items():
            assert torch.equal(t, got[name]), name
    assert p.device_status() == 0
    p.close()


def test_captured_backward_of_an_empty_batch():
    # no kernel of the call before the one that clears the sums
    import torch
    p = _handle(2, 6001, 6, 2)
    p.reserve(1, rk.PASS_SOFT | rk.PASS_BACKWARD)
    X, g = torch.empty((0, 2, 6001), device="cuda"), torch.empty((0, 16), device="cuda")
    arg = torch.empty((0, 8), dtype=torch.int32, device="cuda")
    dW, db = torch.full((p.n_weights,), -7.0, device="cuda"), torch.full((8,), -7.0, device="cuda")
    rk.rocket_transform_soft_backward(p, X, 10.0, 3.0, g, arg, dW, db)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        rk.rocket_transform_soft_backward(p, X, 10.0, 3.0, g, arg, dW, db)
    for _ in range(2):
        dW.fill_(-7)
        db.fill_(-7)
        graph.replay()
        torch.cuda.synchronize()
        assert not dW.any() and not db.any()
    p.close()
