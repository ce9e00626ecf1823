"""Which of the two MINIROCKET kernels serves a call (tests/mini_dispatch_check.cu; nvcc, no GPU): measured shapes, and the cases that
test_gpu_minirocket_kernels.py runs for either of them."""
import os
import subprocess

import pytest

from test_gpu_minirocket_kernels import CASES

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# channels, steps, features, examples; walks
MEASURED = [(250, 10000, 9996, 24, 1), (100, 10000, 840, 24, 1), (20, 10000, 84, 5, 1), (20, 1500, 840, 1, 1), (64, 1500, 840, 1, 1),
            (20, 50000, 9996, 60, 0), (20, 10000, 9996, 24, 0), (1, 512, 9996, 16, 0), (41, 10000, 84, 24, 1), (41, 10000, 4200, 5, 1), (250, 1500, 84, 24, 1), (9, 1500, 4200, 24, 0), (100, 300, 9996, 24, 0)]


def test_dispatch(tmp_path):
    csrc = os.path.join(ROOT, "paper_2301_08527_b200", "csrc")
    exe = str(tmp_path / "mini_dispatch_check")
    subprocess.check_call([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-O1", "-std=c++17",
                           "-I", csrc, "-I", os.path.join(ROOT, "include"), os.path.join(ROOT, "tests", "mini_dispatch_check.cu"), "-o", exe, "-lpthread"])
    rows = MEASURED + [(C, L, F, N, int(walks)) for C, L, N, F, walks in CASES]
    out = subprocess.run([exe], input="".join("%d %d %d %d\n" % r[:4] for r in rows), capture_output=True, text=True, check=True)
    got = list(map(int, out.stdout.split()))
    assert [r for r, g in zip(rows, got) if r[4] != g] == []
