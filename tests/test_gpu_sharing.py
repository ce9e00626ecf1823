"""Small-dilation tiles shared among examples, with a last group that is not full, and series of more than 20 channels on either side of
the line between the fused and the generic kernels, against the oracles (every mode).

Which tiles are shared, and by how many examples, and which kernels serve the series, test_dispatch_host.py checks on the host
for the cases below (buckets of 8 to 31 kernels are class 1, of fewer class 2; 148 SMs).  Served by, for hard, soft and backward: t the tile
kernels, r the one that holds whole examples, g the generic ones.
"""
import numpy as np
import pytest

import oracle
import paper_2301_08527_b200 as rk
from rocket_inputs import ar1_spike_series, normal_array

import parity as P
from test_gpu_edges import _kernels
from test_gpu_f16 import _check_bitwise

# channels, steps, examples, kernels, dilations; classes whose tiles are shared
CASES = [(1, 5003, 103, 60, (1, 2, 9), (1,)), (3, 5002, 83, 40, (1, 2, 3, 5, 6, 7, 11, 13), (2,)),
         (2, 5001, 107, 52, (1, 1, 1, 1, 1, 1, 1, 2, 3, 4, 5, 6, 7), (1, 2)), (4, 5001, 103, 30, (1, 2, 3, 4, 5), (2,))]
# short ones, which share no tiles; served by
SHORT_CASES = [(1, 65, 401, 60, (1, 2, 9), "rrr"), (3, 207, 233, 40, (1, 2, 3, 5, 6, 7, 11, 13), "rrr"),
               (2, 120, 401, 52, (1, 1, 1, 1, 1, 1, 1, 2, 3, 4, 5, 6, 7), "rrr"), (4, 99, 403, 30, (1, 2, 3, 4, 5), "rrr")]
# more than 20 channels; served by
WIDE_CASES = [(21, 1501, 9, 120, (1, 5, 40), "rrr"), (34, 1701, 8, 160, (1, 3, 63, 90), "ttt"), (35, 1500, 8, 160, (2, 9, 130), "rrt"),
              (48, 2003, 6, 90, (1, 2, 7, 66, 160), "ttt"), (25, 86, 3, 60, (1, 2, 5), "rrr"), (255, 130, 5, 40, (1, 4, 9), "rrr"),
              (255, 229, 2, 12, (1, 2, 5, 20), "ggg"), (255, 220, 2, 12, (1, 2, 5, 20), "rrg"), (255, 331, 5, 40, (1, 4, 9), "ttt")]


def kernels(C, L, K, dilations):
    return _kernels(np.random.default_rng(1000 * C + L), C, L, K, dilations, 9)


@pytest.mark.gpu
@pytest.mark.parametrize("case", CASES + SHORT_CASES + WIDE_CASES)
def test_every_mode(case):
    import torch
    C, L, N, K, dilations, _ = case
    kp = kernels(C, L, K, dilations)
    X = ar1_spike_series(C + L, N, C, L)
    lam, shift = 10.0, 3.0
    p = rk.RocketParams.from_kernel_params(kp)
    Xd = torch.from_numpy(X).cuda()
    ref = oracle.forward(kp, X, lam=lam, shift=shift)
    ppv, mx = P.split_features(rk.rocket_transform(p, Xd).cpu().numpy())
    P.check_hard_ppv(ppv, ref)
    P.check_max(mx, ref)
    if C <= 20:
        _check_bitwise(kp, X, rk.rocket_transform_f16(p, Xd).cpu().numpy())
    feat, arg = rk.rocket_transform_soft(p, Xd, lam, shift)
    soft, mx = P.split_features(feat.cpu().numpy())
    P.check_soft_ppv(soft, ref)
    P.check_max(mx, ref)
    P.check_argmax(arg.cpu().numpy(), ref)
    g = normal_array(L, (N, 2 * kp.K))
    dW, db = rk.rocket_transform_soft_backward(p, Xd, lam, shift, torch.from_numpy(g).cuda(), arg)
    rW, rb = oracle.backward(kp, X, g, arg.cpu().numpy(), lam=lam, shift=shift)
    P.check_grads(dW.cpu().numpy(), db.cpu().numpy(), rW, rb)
    assert p.device_status() == 0
    p.close()


@pytest.mark.gpu
@pytest.mark.parametrize("C,L,K,N", [(255, 4000, 60, 32), (32, 301, 1500, 40), (21, 33, 1500, 64)])
def test_a_call_covers_the_smaller_ones_of_its_kind(C, L, K, N):
    # whichever kernels serve them: no call allocates after a larger one
    import torch
    p = rk.RocketParams.generate(8527, K, C, L)
    X = torch.from_numpy(ar1_spike_series(C + L, N, C, L)).cuda()
    g = torch.from_numpy(normal_array(L, (N, 2 * K))).cuda()

    def calls(n):
        rk.rocket_transform(p, X[:n])
        _, arg = rk.rocket_transform_soft(p, X[:n], 10.0, 3.0)
        return rk.rocket_transform_soft_backward(p, X[:n], 10.0, 3.0, g[:n].contiguous(), arg)

    calls(N)
    before = rk.device_alloc_count()
    for n in [*range(1, N, 3), N]:
        calls(n)
    torch.cuda.synchronize()
    assert rk.device_alloc_count() == before
    p.close()
