"""rocket_params_reserve: after it, device calls within the reserved size allocate nothing."""
import numpy as np
import pytest

import oracle
import paper_2301_08527_b200 as rk
from rocket_inputs import ar1_spike_series, generate_kernels, kernels_from_lists, normal_array

import parity as P

pytestmark = pytest.mark.gpu


def _kernels_with_generic_lengths(C, L):
    rng = np.random.default_rng(5)
    ks = []
    for i in range(60):
        ln = [3, 5, 7, 9, 11][i % 5]
        d = int(rng.integers(1, max(2, (L - 1) // (ln - 1) // 2)))
        ks.append(dict(dilation=d, padding=(ln - 1) * d // 2 if i % 2 else 0, channels=sorted(rng.choice(C, 2, replace=False).tolist()),
                       weights=rng.normal(size=(2, ln)), bias=float(rng.uniform(-1, 1))))
    return kernels_from_lists(C, L, ks)


@pytest.mark.parametrize("case", ["fused kernels only", "fused and generic kernels", "generic path"])
def test_calls_after_reserve_do_not_allocate(case):
    import torch
    C, L, N = 6, 4000, 30                      # one pass of the fused kernels
    kp = generate_kernels(91, 400, C, L) if case != "fused and generic kernels" else _kernels_with_generic_lengths(C, L)
    X = ar1_spike_series(92, N, C, L)
    g = normal_array(93, (N, 2 * kp.K))
    Xd = torch.from_numpy(X).cuda()
    gd = torch.from_numpy(g).cuda()
    X8 = torch.from_numpy(np.clip(np.round(X * 40 + 128), 0, 255).astype(np.uint8)).cuda()
    mean, istd = np.full(C, 128.0, np.float32), np.full(C, 1 / 40.0, np.float32)
    p = rk.RocketParams.from_kernel_params(kp)
    if case == "generic path":
        p.set_path(1)
    feat = torch.empty((N, 2 * kp.K), device="cuda")
    arg = torch.empty((N, kp.K), dtype=torch.int32, device="cuda")
    dW = torch.empty((p.n_weights,), device="cuda")
    db = torch.empty((kp.K,), device="cuda")
    p.reserve(N, rk.PASS_HARD | rk.PASS_SOFT | rk.PASS_BACKWARD | rk.PASS_U8_INPUT)
    torch.cuda.synchronize()
    before = rk.device_alloc_count()
    for n in (N, 7, N):                                     # smaller calls fit as well
        rk.rocket_transform(p, Xd[:n], out=feat[:n])
        rk.rocket_transform_soft(p, Xd[:n], 10.0, 3.0, out=feat[:n], argmax_out=arg[:n])
        rk.rocket_transform_soft_backward(p, Xd[:n], 10.0, 3.0, gd[:n], arg[:n], dW, db)
        rk.rocket_transform_u8(p, X8[:n], mean, istd, out=feat[:n])
    torch.cuda.synchronize()
    assert rk.device_alloc_count() == before, "a device call allocated after rocket_params_reserve"
    assert p.device_status() == 0
    # and the reserved workspace gives the right answers
    ref = oracle.forward(kp, X, lam=10.0, shift=3.0)
    sfeat, sarg = rk.rocket_transform_soft(p, Xd, 10.0, 3.0)
    soft, mx = P.split_features(sfeat.cpu().numpy())
    P.check_soft_ppv(soft, ref)
    P.check_max(mx, ref)
    dW2, db2 = rk.rocket_transform_soft_backward(p, Xd, 10.0, 3.0, gd, torch.from_numpy(ref.argmax.astype(np.int32)).cuda())
    rdW, rdb = oracle.backward(kp, X, g, ref.argmax, lam=10.0, shift=3.0)
    P.check_grads(dW2.cpu().numpy(), db2.cpu().numpy(), rdW, rdb)
    # a larger call than reserved still works (and may allocate)
    p.reserve(N + 5, rk.PASS_HARD)
    p.close()


def test_fused_and_generic_kernels_in_several_passes():
    # 800 MB of staging copies hold 13 examples of 20 x 50,000
    import torch
    C, L, N = 20, 50000, 28
    rng = np.random.default_rng(6)
    ks = []
    for i in range(25):
        ln = [3, 5, 7, 9, 11][i % 5]
        d = [1, 9, 61, 300, 3001][i // 5]
        ks.append(dict(dilation=d, padding=(ln - 1) * d // 2 if i % 2 else 0, channels=sorted(rng.choice(C, 2, replace=False).tolist()),
                       weights=rng.normal(size=(2, ln)), bias=float(rng.uniform(-1, 1))))
    ks.append(dict(dilation=8333, padding=0, channels=[3], weights=rng.normal(size=(1, 7)), bias=0.1))    # widest margins of the copies
    kp = kernels_from_lists(C, L, ks)
    X = np.tile(ar1_spike_series(95, 4, C, L), (7, 1, 1))
    g = normal_array(96, (N, 2 * kp.K))
    Xd, gd = torch.from_numpy(X).cuda(), torch.from_numpy(g).cuda()
    p = rk.RocketParams.from_kernel_params(kp)
    p.reserve(N, rk.PASS_HARD | rk.PASS_SOFT | rk.PASS_BACKWARD)
    before, launches = rk.device_alloc_count(), rk.kernel_launch_count()
    ppv, mx = P.split_features(rk.rocket_transform(p, Xd).cpu().numpy())
    many = rk.kernel_launch_count() - launches
    rk.rocket_transform(p, Xd[:2])
    assert many - (rk.kernel_launch_count() - launches - many) >= 2 * 3, "copy and both fused kernels of at least two more passes"
    feat, arg = rk.rocket_transform_soft(p, Xd, 10.0, 3.0)
    dW, db = rk.rocket_transform_soft_backward(p, Xd, 10.0, 3.0, gd, arg)
    torch.cuda.synchronize()
    assert rk.device_alloc_count() == before
    ref = oracle.forward(kp, X[:4], lam=10.0, shift=3.0)
    soft, smx = P.split_features(feat.cpu().numpy())
    for n0 in range(0, N, 4):                               # the same four examples over and over
        P.check_hard_ppv(ppv[n0:n0 + 4], ref)
        P.check_max(mx[n0:n0 + 4], ref)
        P.check_soft_ppv(soft[n0:n0 + 4], ref)
        P.check_max(smx[n0:n0 + 4], ref)
        P.check_argmax(arg[n0:n0 + 4].cpu().numpy(), ref)
    arg = arg.cpu().numpy()
    assert np.array_equal(arg, np.tile(arg[:4], (7, 1)))
    # linear in the incoming gradient: that of the seven copies of an example is their sum's
    rW, rb = oracle.backward(kp, X[:4], g.reshape(7, 4, -1).sum(0).astype(np.float32), arg[:4], lam=10.0, shift=3.0)
    P.check_grads(dW.cpu().numpy(), db.cpu().numpy(), rW, rb)
    assert p.device_status() == 0
    p.close()


def test_reserve_rejects_bad_arguments():
    kp = generate_kernels(94, 20, 2, 200)
    p = rk.RocketParams.from_kernel_params(kp)
    lib = rk.load_library()
    assert lib.rocket_params_reserve(p.handle, 0, 1) == -1
    assert lib.rocket_params_reserve(p.handle, 4, 0) == -1
    assert lib.rocket_params_reserve(p.handle, 4, 16) == -1
    assert lib.rocket_params_reserve(None, 4, 1) == -1
    p.close()
