"""Host checks of the dispatch rules (tests/dispatch_check.cpp)."""
import os
import subprocess

import pytest

from test_gpu_sharing import CASES, SHORT_CASES, WIDE_CASES, kernels

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    csrc = os.path.join(ROOT, "paper_2301_08527_b200", "csrc")
    exe = str(tmp_path_factory.mktemp("dispatch") / "dispatch_check")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I", csrc, "-I", os.path.join(ROOT, "include"), "-I", "/usr/local/cuda/include",
                           os.path.join(ROOT, "tests", "dispatch_check.cpp"), os.path.join(csrc, "rocket_plan.cpp"),
                           os.path.join(csrc, "rocket_generate.cpp"), "-o", exe])
    return exe


def test_dispatch_rules(check):
    out = subprocess.run([check], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr


def _dispatch(check, C, L, N, kp):
    """(examples that share a tile, tiles) per class, and which kernels serve the call in each mode."""
    text = "%d %d %d\n" % (C, L, kp.K)
    for k in range(kp.K):
        ch = kp.channel_idx[kp.channel_offset[k]:kp.channel_offset[k + 1]]
        text += " ".join(map(str, [kp.length[k], kp.dilation[k], kp.padding[k], len(ch), *ch])) + "\n"
    out = subprocess.run([check, str(N)], input=text, capture_output=True, text=True, check=True).stdout.split()
    return list(map(int, out[0:6:2])), list(map(int, out[1:6:2])), out[6]


@pytest.mark.parametrize("case", CASES)
def test_the_sharing_cases_share_tiles(check, case):
    C, L, N, K, dilations, classes = case
    examples, tiles, served = _dispatch(check, C, L, N, kernels(C, L, K, dilations))
    assert served == "ttt"
    for cls in classes:
        assert tiles[cls] > 0 and examples[cls] > 1 and N % examples[cls] != 0, (examples, tiles)


@pytest.mark.parametrize("case", SHORT_CASES + WIDE_CASES)
def test_the_other_cases_take_the_kernels_they_name(check, case):
    C, L, N, K, dilations, served = case
    assert _dispatch(check, C, L, N, kernels(C, L, K, dilations))[2] == served
