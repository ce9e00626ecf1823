"""The failure flag of a MINIROCKET call, and batches that take several launches (tests/mini_flag_check.cu)."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _run(tmp_path, name, *defines):
    csrc = os.path.join(ROOT, "paper_2301_08527_b200", "csrc")
    exe = str(tmp_path / name)
    subprocess.check_call([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-O1", "-std=c++17",
                           "-I", csrc, "-I", os.path.join(ROOT, "include"), os.path.join(ROOT, "tests", "mini_flag_check.cu"), "-o", exe, "-lpthread",
                           *defines])
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout + out.stderr
    return out.stdout


def test_a_failed_wait_marks_its_own_call_only(tmp_path):
    _run(tmp_path, "whole")


def test_a_batch_in_several_launches_gives_the_same_bits(tmp_path):
    # 50 examples, 7 and 1 per launch
    whole = _run(tmp_path, "whole")
    assert _run(tmp_path, "seven", "-DROCKET_MINI_LAUNCH_TILES=(7 * n_tiles)") == whole
    assert _run(tmp_path, "one", "-DROCKET_MINI_LAUNCH_TILES=1") == whole
