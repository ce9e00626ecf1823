"""The reciprocal that the ridge factorisation divides by, against correctly rounded quotients (tests/reciprocal_check.cu)."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_quotients_by_way_of_the_reciprocal(tmp_path):
    exe = str(tmp_path / "reciprocal_check")
    subprocess.check_call([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17",
                           "-I", os.path.join(ROOT, "paper_2301_08527_b200", "csrc"), os.path.join(ROOT, "tests", "reciprocal_check.cu"), "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout + out.stderr
    print(out.stdout)
