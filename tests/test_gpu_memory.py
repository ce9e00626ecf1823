"""Handles whose staging copies do not fit the device: smaller parts of the batch, then the generic kernels, and the same results."""
import numpy as np
import pytest

import paper_2301_08527_b200 as rk
from rocket_inputs import ar1_spike_series, kernels_from_lists, normal_array

pytestmark = pytest.mark.gpu


def _leave(room):
    """Takes the device's memory but for `room` bytes."""
    import torch
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    return torch.empty(max(0, free - room), dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("C", [6, 30])
def test_less_memory_than_the_copies_take(C):
    import torch
    L, N, K = 60000, 12, 12
    rng = np.random.default_rng(C)
    ks = [dict(dilation=[1, 5, 70, 300, 1001, 4003][i % 6], padding=0, channels=sorted(rng.choice(C, 3, replace=False).tolist()),
               weights=rng.normal(size=(3, (7, 9, 11)[i % 3])), bias=float(rng.uniform(-1, 1))) for i in range(K)]
    kp = kernels_from_lists(C, L, ks)
    X = torch.from_numpy(np.tile(ar1_spike_series(C, 3, C, L), (4, 1, 1))).cuda()
    g = torch.from_numpy(normal_array(5, (N, 2 * K))).cuda()

    def buffers(p):
        return {"hard": torch.empty((N, 2 * K), device="cuda"), "soft": torch.empty((N, 2 * K), device="cuda"),
                "arg": torch.empty((N, K), dtype=torch.int32, device="cuda"), "dW": torch.empty(p.n_weights, device="cuda"),
                "db": torch.empty(K, device="cuda")}

    def run(p, out):
        rk.rocket_transform(p, X, out=out["hard"])
        rk.rocket_transform_soft(p, X, 10.0, 3.0, out=out["soft"], argmax_out=out["arg"])
        rk.rocket_transform_soft_backward(p, X, 10.0, 3.0, g, out["arg"], out["dW"], out["db"])
        torch.cuda.synchronize()
        return out

    p = rk.RocketParams.from_kernel_params(kp)
    want = run(p, buffers(p))
    p.close()
    example = 28 * C * (L + 7 * 4003)                      # one example's copies
    for room, exact in ((int(4.5 * example), True), (example // 2, False)):
        p = rk.RocketParams.from_kernel_params(kp)
        p.bind_device()
        first, second, third = buffers(p), buffers(p), buffers(p)
        held = _leave(room + (8 << 20))                    # besides: the workspaces of the soft passes
        got = run(p, first)
        before = rk.device_alloc_count()
        again = run(p, second)
        assert rk.device_alloc_count() == before, "the allocation that failed is tried again"
        assert p.device_status() == 0
        del held
        torch.cuda.empty_cache()
        for name, t in want.items():
            assert torch.equal(got[name], again[name]), name
            if exact and name in ("hard", "soft", "arg"):
                assert torch.equal(t, got[name]), name
            else:                                          # sums in another order
                err = (t.double() - got[name].double()).norm() / t.double().norm()
                assert err <= 1e-5, (name, float(err))
        p.reserve(N, rk.PASS_HARD | rk.PASS_SOFT | rk.PASS_BACKWARD)   # there is room now
        full = run(p, third)
        for name in ("hard", "soft", "arg"):
            assert torch.equal(want[name], full[name]), name
        p.close()


def _fit_problem(N, P):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(N)
    F = torch.rand((N, P), generator=g, device="cuda")
    return F, torch.randn((N,), generator=g, device="cuda")


def _give_back():
    """The regressor's workspace goes when a handle does."""
    p = rk.RocketParams.generate(1, 1, 1, 64)
    p.bind_device()
    p.close()


def test_a_fit_goes_on_without_room_for_the_features_as_integers():
    import torch
    F, y = _fit_problem(677, 20000)
    want, _ = rk.rocket_ridge_fit(F, y, 1.0)
    _give_back()
    held = _leave(64 << 20)                                # the digits alone take 107 MB, all the rest 45
    got, _ = rk.rocket_ridge_fit(F, y, 1.0)
    del held
    torch.cuda.empty_cache()
    # both as close as double precision goes: rounded to FP32 each
    assert (got.double() - want.double()).norm() <= 2.0 ** -23 * want.double().norm()
    _give_back()


def test_larger_fits_keep_their_workspace_too():
    F, y = _fit_problem(1600, 20000)
    rk.rocket_ridge_fit(F, y, 1.0)
    before = rk.device_alloc_count()
    rk.rocket_ridge_fit(F, y, 1.0)
    assert rk.device_alloc_count() == before
    _give_back()
