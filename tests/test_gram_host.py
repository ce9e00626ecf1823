"""Host check of the plan of the integer Gram matrix (tests/gram_check.cpp)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_slice_of_every_chunk_has_columns(tmp_path):
    csrc = os.path.join(ROOT, "paper_2301_08527_b200", "csrc")
    exe = str(tmp_path / "gram_check")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I", csrc, "-I", "/usr/local/cuda/include", os.path.join(ROOT, "tests", "gram_check.cpp"),
                           "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
