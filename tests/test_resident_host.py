"""Host check of the resident kernel's plan (tests/resident_check.cpp)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_output_is_owned_once_and_reads_stay_in_the_series(tmp_path):
    csrc = os.path.join(ROOT, "paper_2301_08527_b200", "csrc")
    exe = str(tmp_path / "resident_check")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I", csrc, "-I", os.path.join(ROOT, "include"), "-I", "/usr/local/cuda/include",
                           os.path.join(ROOT, "tests", "resident_check.cpp"), os.path.join(csrc, "rocket_plan.cpp"),
                           os.path.join(csrc, "rocket_generate.cpp"), "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
