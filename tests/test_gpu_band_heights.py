"""Small-dilation tiles of 24, 21 and 18 rows: the plan's coverage (tests/height_check.cpp) and every mode against the oracles."""
import os
import subprocess

import numpy as np
import pytest

import oracle
import paper_2301_08527_b200 as rk
from rocket_inputs import ar1_spike_series, normal_array

import parity as P
from test_gpu_edges import _kernels
from test_gpu_f16 import _check_bitwise

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
# channels, steps, examples, rows of a band; dilations 1 to 13
CASES = [(20, 3207, 2, 18), (20, 3300, 2, 18), (20, 3601, 2, 21), (20, 4800, 2, 21), (20, 4001, 2, 24)]


def _handle(C, L):
    return _kernels(np.random.default_rng(C * L), C, L, 40, (1, 2, 3, 5, 8, 13), 5)


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    csrc = os.path.join(ROOT, "paper_2301_08527_b200", "csrc")
    exe = str(tmp_path_factory.mktemp("heights") / "height_check")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I", csrc, "-I", os.path.join(ROOT, "include"), "-I", "/usr/local/cuda/include",
                           os.path.join(ROOT, "tests", "height_check.cpp"), os.path.join(csrc, "rocket_plan.cpp"),
                           os.path.join(csrc, "rocket_generate.cpp"), "-o", exe])
    return exe


def test_every_output_is_owned_once(check):
    out = subprocess.run([check], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr


@pytest.mark.parametrize("C,L,N,rows", CASES)
def test_the_cases_take_the_height_they_name(check, C, L, N, rows):
    kp = _handle(C, L)
    text = "%d\n" % kp.K
    for k in range(kp.K):
        ch = kp.channel_idx[kp.channel_offset[k]:kp.channel_offset[k + 1]]
        text += " ".join(map(str, [kp.length[k], kp.dilation[k], kp.padding[k], len(ch), *ch])) + "\n"
    out = subprocess.run([check, str(C), str(L)], input=text, capture_output=True, text=True, check=True).stdout.split()
    assert out == [str(rows), "0"]


@pytest.mark.gpu
@pytest.mark.parametrize("C,L,N,rows", CASES)
def test_every_mode(C, L, N, rows):
    import torch
    kp = _handle(C, L)
    X = ar1_spike_series(L, N, C, L)
    lam, shift = 10.0, 3.0
    p = rk.RocketParams.from_kernel_params(kp)
    Xd = torch.from_numpy(X).cuda()
    ref = oracle.forward(kp, X, lam=lam, shift=shift)
    ppv, mx = P.split_features(rk.rocket_transform(p, Xd).cpu().numpy())
    P.check_hard_ppv(ppv, ref)
    P.check_max(mx, ref)
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
