"""The kernel that holds whole examples in shared memory, at the edges of its tiles and of its range, against the oracles (every mode).

Rows of a dilation around multiples of its bands of 5 to 21 rows (one height or two), columns around the 64 of a tile, examples that fill shared memory with no room
for zeros between the rows, samples at odd addresses, one more step than it serves, more examples than blocks, one kernel.  Tiles shared
among examples (small dilations of the other kernels) at a length beyond this kernel's.
"""
import numpy as np
import pytest

import oracle
import paper_2301_08527_b200 as rk
from rocket_inputs import ar1_spike_series, channel_statistics, intensity_series_u8, normal_array

import parity as P
from test_gpu_edges import _kernels
from test_gpu_f16 import _check_bitwise

pytestmark = pytest.mark.gpu

# channels, steps, examples, kernels, dilations
CASES = [(1, 64, 3, 24, (1, 2, 3, 5, 7)), (2, 152, 5, 30, (8, 9, 15, 16, 17)), (3, 153, 4, 30, (1, 2, 4, 8, 9, 17)), (5, 1088, 2, 40, (1, 3, 31, 32, 33, 63, 64, 65)),
         (1, 1089, 149, 12, (1, 2, 100)), (32, 1800, 2, 30, (1, 2, 7, 40, 128, 179)), (28, 2047, 2, 24, (1, 6, 65, 200)), (7, 301, 300, 1, (4,)),
         (6, 640, 3, 30, (1, 2, 5, 11, 60, 106)), (4, 900, 3, 30, (1, 3, 14, 15, 16, 149)), (3, 1344, 4, 30, (1, 2, 21, 63, 64, 223)),
         (2, 1409, 3, 30, (1, 2, 11, 64, 65, 234)), (20, 1251, 2, 24, (1, 2, 30, 208)), (1, 5000, 2, 24, (1, 2, 9, 70, 400)), (1, 5001, 2, 24, (1, 2, 9, 70, 400)), (2, 6001, 41, 20, (1, 2, 3, 11))]


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("C,L,N,K,dilations", CASES)
def test_every_mode(C, L, N, K, dilations, shift):
    import torch
    kp = _kernels(np.random.default_rng(C + L), C, L, K, dilations, 9)
    X = ar1_spike_series(C * L, N, C, L)
    lam, sh = 10.0, 3.0
    p = rk.RocketParams.from_kernel_params(kp)
    room = torch.zeros(X.size + shift, device="cuda")
    Xd = room[shift:].view(N, C, L)                        # at an odd multiple of four bytes for shift = 1
    Xd.copy_(torch.from_numpy(X))
    ref = oracle.forward(kp, X, lam=lam, shift=sh)
    ppv, mx = P.split_features(rk.rocket_transform(p, Xd).cpu().numpy())
    P.check_hard_ppv(ppv, ref)
    P.check_max(mx, ref)
    if C <= 20:
        _check_bitwise(kp, X, rk.rocket_transform_f16(p, Xd).cpu().numpy())
    feat, arg = rk.rocket_transform_soft(p, Xd, lam, sh)
    soft, mx = P.split_features(feat.cpu().numpy())
    P.check_soft_ppv(soft, ref)
    P.check_max(mx, ref)
    P.check_argmax(arg.cpu().numpy(), ref)
    g = normal_array(L, (N, 2 * K))
    dW, db = rk.rocket_transform_soft_backward(p, Xd, lam, sh, torch.from_numpy(g).cuda(), arg)
    rW, rb = oracle.backward(kp, X, g, arg.cpu().numpy(), lam=lam, shift=sh)
    P.check_grads(dW.cpu().numpy(), db.cpu().numpy(), rW, rb)
    assert p.device_status() == 0
    p.close()


def test_bytes_give_the_bits_of_their_samples():
    import torch
    C, L, N, K = 6, 1252, 9, 60
    kp = _kernels(np.random.default_rng(3), C, L, K, (1, 2, 5, 33, 90), 5)
    X8 = intensity_series_u8(4, N, C, L)
    mean, inv_std = channel_statistics(X8)
    p = rk.RocketParams.from_kernel_params(kp)
    got = rk.rocket_transform_u8(p, torch.from_numpy(X8).cuda(), mean, inv_std)
    scaled = (torch.from_numpy(X8).cuda().float() - torch.from_numpy(mean).cuda().view(1, -1, 1)) * torch.from_numpy(inv_std).cuda().view(1, -1, 1)
    want = rk.rocket_transform(p, scaled.contiguous())
    assert torch.equal(got, want)
    p.close()


def _many_kernels(C, L, K):
    import torch
    p = rk.RocketParams.generate(8527, K, C, L)
    return p, lambda N: torch.from_numpy(np.tile(ar1_spike_series(C, 8, C, L), (-(-N // 8), 1, 1))[:N].copy()).cuda()


def _launches(call):
    before = rk.kernel_launch_count()
    out = call()
    return rk.kernel_launch_count() - before, out


def test_large_hard_transforms_take_the_tile_kernels():
    # from 6e5 (kernel, example) pairs on beyond 2,048 steps; the same bits, one example more or less, and the other modes stay
    import torch
    C, L, K = 3, 2100, 10000
    p, series = _many_kernels(C, L, K)
    X = series(60)
    n, large = _launches(lambda: rk.rocket_transform(p, X))
    assert n > 1
    n, small = _launches(lambda: rk.rocket_transform(p, X[:59].contiguous()))
    assert n == 1
    assert torch.equal(large[:59], small)
    assert _launches(lambda: rk.rocket_transform_f16(p, X))[0] == 1
    assert _launches(lambda: rk.rocket_transform_soft(p, X, 10.0, 3.0))[0] == 1
    v = ((X - X.min()) * (255 / (X.max() - X.min()))).to(torch.uint8)
    mean, inv_std = np.full(C, 100.0, np.float32), np.full(C, 1 / 40.0, np.float32)
    n, large = _launches(lambda: rk.rocket_transform_u8(p, v, mean, inv_std))
    assert n > 1
    assert torch.equal(large[:59], rk.rocket_transform_u8(p, v[:59].contiguous(), mean, inv_std))
    assert p.device_status() == 0
    p.close()


def test_large_hard_transforms_after_reserve_and_without_it():
    import torch
    C, L, K = 3, 2100, 10000
    p, series = _many_kernels(C, L, K)
    X = series(64)
    p.reserve(64, rk.PASS_HARD)
    before = rk.device_alloc_count()
    n, want = _launches(lambda: rk.rocket_transform(p, X))
    assert n > 1 and rk.device_alloc_count() == before
    p.close()
    # nothing reserved: a capture goes on, with the kernel that needs no workspace
    p, _ = _many_kernels(C, L, K)
    rk.rocket_transform(p, X[:1].contiguous())
    out = torch.zeros_like(want)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        rk.rocket_transform(p, X, out=out)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    del graph
    p.close()
    # next to no room: fewer examples at a time, or that kernel
    p, _ = _many_kernels(C, L, K)
    p.bind_device()
    torch.cuda.empty_cache()
    held = torch.empty(max(0, torch.cuda.mem_get_info()[0] - (4 << 20)), dtype=torch.uint8, device="cuda")
    rk.rocket_transform(p, X, out=out.zero_())
    torch.cuda.synchronize()
    del held
    torch.cuda.empty_cache()
    assert torch.equal(out, want)
    p.close()
