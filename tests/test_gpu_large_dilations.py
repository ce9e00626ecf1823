"""Handles with dilations beyond (2 L + 4096) / 7, which the kernel on four staging copies serves: every mode against the oracles.

Such a dilation takes a padding that brings the output range to at least one output.  Kernels of small and of ordinary large
dilations are in the same handle, so that both fused kernels of a pass run.
"""
import numpy as np
import pytest

import oracle
import paper_2301_08527_b200 as rk
from rocket_inputs import ar1_spike_series, channel_statistics, intensity_series_u8, kernels_from_lists, normal_array

import parity as P
from test_gpu_f16 import _check_bitwise

pytestmark = pytest.mark.gpu


def _kernels(C, L, K, seed):
    rng = np.random.default_rng(seed)
    least = (2 * L + 4096) // 7 + 1
    ks = []
    for i in range(K):
        ln = (7, 9, 11)[i % 3]
        kind = i % 5
        if kind == 0:
            d = int(rng.integers(1, 60))
        elif kind == 1:
            d = int(rng.integers(64, max(65, (L - 1) // (ln - 1))))
        else:
            d = int(rng.integers(least, 2 * least)) // 4 * 4 + i % 4      # every residue modulo four
            d = max(d, least)
        span = (ln - 1) * d
        lowest = max(0, (span - L) // 2 + 1)
        p = [span // 2, lowest, max(lowest, span // 2 + 17), max(lowest, span)][int(rng.integers(0, 4))]
        m = int(rng.integers(1, min(C, ln, 5) + 1))
        ks.append(dict(dilation=d, padding=int(p), channels=sorted(rng.choice(C, m, replace=False).tolist()), weights=rng.normal(size=(m, ln)),
                       bias=float(rng.uniform(-1, 1))))
    kp = kernels_from_lists(C, L, ks)
    assert 7 * int(kp.dilation.max()) > 2 * L + 4096
    return kp


@pytest.mark.parametrize("C,L,N,K", [(1, 300, 3, 30), (3, 1001, 4, 45), (20, 3000, 2, 40), (30, 2003, 2, 40), (5, 12004, 3, 30)])
def test_every_mode(C, L, N, K):
    import torch
    kp = _kernels(C, L, K, seed=C + L)
    X = ar1_spike_series(L, N, C, L)
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


@pytest.mark.parametrize("C,L,N,K", [(3, 1000, 4, 45), (20, 3000, 2, 40)])
def test_bytes(C, L, N, K):
    import torch
    kp = _kernels(C, L, K, seed=C + L + 1)
    X8 = intensity_series_u8(L, N, C, L)
    mean, inv_std = channel_statistics(X8)
    p = rk.RocketParams.from_kernel_params(kp)
    ref = oracle.forward(kp, oracle.scale_u8(X8, mean, inv_std))
    ppv, mx = P.split_features(rk.rocket_transform_u8(p, torch.from_numpy(X8).cuda(), mean, inv_std).cpu().numpy())
    P.check_hard_ppv(ppv, ref)
    P.check_max(mx, ref)
    assert p.device_status() == 0
    p.close()
