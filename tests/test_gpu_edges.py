"""Where the dispatch of the fused kernels changes, against the oracle with the tolerances of parity.py.

Small dilations: 20, 21, 34 and 35 channels in one dilation (one bucket; halves of a tile; halves with every plane in use; several
buckets); light buckets that share a tile among examples, with a last group that is not full.  Large dilations: every residue of
the dilation modulo four (rows per step of a bulk copy), dilations around a multiple of the tile's 64 columns, output ranges that end
in bands of 16, 12 and 8 rows.  MINIROCKET: 20, 21, 40 and 41 channels in one dilation (two tiles in shared memory; one large
tile, full; several buckets), fewer samples than a tile has columns.  Ridge: more examples than a block takes, feature counts around
the width of its loads, rows that start at odd addresses.
"""
import numpy as np
import pytest

import oracle
import paper_2301_08527_b200 as rk
from rocket_inputs import ar1_spike_series, kernels_from_lists, normal_array

import parity as P
from test_gpu_minirocket import _check as check_minirocket
from test_gpu_ridge import _dev, _problem

pytestmark = pytest.mark.gpu


def _kernels(rng, C, L, K, dilations, most_channels):
    ks = []
    for i in range(K):
        d = int(dilations[i % len(dilations)])
        ln = int(rng.choice([n for n in (7, 9, 11) if (n - 1) * d < L]))
        m = int(rng.integers(1, min(C, ln, most_channels) + 1))
        ks.append(dict(dilation=d, padding=(ln - 1) * d // 2 if rng.random() < 0.5 else 0, channels=sorted(rng.choice(C, m, replace=False).tolist()),
                       weights=rng.normal(size=(m, ln)), bias=float(rng.uniform(-1, 1))))
    return kernels_from_lists(C, L, ks)


@pytest.mark.parametrize("C,L,N,K,dilations", [
    (20, 301, 3, 60, (1, 5, 40)), (21, 301, 3, 60, (1, 5, 40)), (34, 1001, 2, 120, (1, 3, 63)), (35, 700, 2, 90, (2, 9)),
    (3, 207, 17, 40, (1, 2, 3, 5, 6, 7, 11, 13)), (1, 65, 33, 12, (1, 2, 9)),
    (3, 2403, 2, 48, (64, 65, 66, 67, 126, 127, 128, 129)), (4, 5002, 3, 40, (191, 193, 254, 301, 500, 601, 703, 829)),
])
def test_transforms_and_backward(C, L, N, K, dilations):
    import torch
    rng = np.random.default_rng(1000 * C + L)
    kp = _kernels(rng, C, L, K, dilations, 9)
    X = ar1_spike_series(C + L, N, C, L)
    lam, shift = 10.0, 3.0
    p = rk.RocketParams.from_kernel_params(kp)
    Xd = torch.from_numpy(X).cuda()
    ref = oracle.forward(kp, X, lam=lam, shift=shift)
    ppv, mx = P.split_features(rk.rocket_transform(p, Xd).cpu().numpy())
    P.check_hard_ppv(ppv, ref)
    P.check_max(mx, ref)
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


@pytest.mark.parametrize("C,L,N,F", [(20, 331, 3, 84 * 5), (21, 331, 3, 84 * 5), (40, 1203, 2, 84 * 9), (41, 500, 2, 84 * 6), (32, 33, 2, 84)])
def test_minirocket(C, L, N, F):
    check_minirocket(C, L, N, F, seed=500 + C)


@pytest.mark.parametrize("N,P_,offset", [(1, 4, 0), (3, 1025, 0), (65, 128, 1), (130, 4099, 3), (300, 31, 2)])
def test_ridge_predict(N, P_, offset):
    # a sum of P products of order one in fp32 (partial sums over the threads of a block): 2e-6 of the scale of the terms
    F, y = _problem(N + P_, N, P_)
    w = np.random.default_rng(P_).normal(0, 1.0 / np.sqrt(P_), P_).astype(np.float32)
    import torch
    raw = torch.zeros(N * P_ + offset, device="cuda")
    raw[offset:] = _dev(F).reshape(-1)
    got = rk.rocket_ridge_predict(raw[offset:].view(N, P_), _dev(w), _dev(np.array([1.2], np.float32))).cpu().numpy()
    want = F.astype(np.float64) @ w.astype(np.float64) + np.float32(1.2)
    assert np.abs(got - want).max() <= 2e-6 * max(1.0, float(np.abs(want).max()), float((np.abs(F) @ np.abs(w)).max()))


@pytest.mark.parametrize("N,P_", [(70, 4100), (3, 8196), (37, 16388), (1, 20000), (148, 4096), (149, 4100)])
def test_ridge_predict_rows_shared_by_a_cluster(N, P_):
    # rows of whole 16-byte loads shared by 2, 4 and 8 blocks, in parts that are not of one size; 148 rows are the most that
    # two blocks share
    F, y = _problem(N + P_, N, P_)
    w = np.random.default_rng(P_).normal(0, 1.0 / np.sqrt(P_), P_).astype(np.float32)
    got = [rk.rocket_ridge_predict(_dev(F), _dev(w), _dev(np.array([1.2], np.float32))).cpu().numpy() for _ in range(20)]
    want = F.astype(np.float64) @ w.astype(np.float64) + np.float32(1.2)
    # summed in double and rounded once: half a unit of the result, and the double sum's own error far below that
    assert np.abs(got[0] - want).max() <= 1.2e-7 * max(1.0, float(np.abs(want).max()))
    assert all(np.array_equal(g, got[0]) for g in got)


@pytest.mark.parametrize("N,P_,offset", [(299, 127, 0), (300, 128, 0), (600, 256, 0), (599, 256, 0), (1201, 512, 0), (301, 31, 1), (600, 33, 3),
                                         (70001, 5, 0), (66000, 64, 0), (149, 6144, 0), (148, 6145, 1), (7, 1023, 0), (9, 4100, 0),
                                         (2000, 897, 0), (2001, 4092, 0), (2001, 2049, 2)])
def test_ridge_predict_of_many_rows(N, P_, offset):
    # a warp (one load per lane, or many rows), half a block and a block per row, at the edges between them and in both widths of load
    rng = np.random.default_rng(N + P_)
    F = rng.normal(0.5, 1.0, (N, P_)).astype(np.float32)
    w = rng.normal(0, 1.0 / np.sqrt(P_), P_).astype(np.float32)
    import torch
    raw = torch.zeros(N * P_ + offset, device="cuda")
    raw[offset:] = _dev(F).reshape(-1)
    got = rk.rocket_ridge_predict(raw[offset:].view(N, P_), _dev(w), _dev(np.array([1.2], np.float32))).cpu().numpy()
    want = F.astype(np.float64) @ w.astype(np.float64) + np.float32(1.2)
    assert np.abs(got - want).max() <= 1.2e-7 * max(1.0, float(np.abs(want).max()))   # summed in double, rounded once
