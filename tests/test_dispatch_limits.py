"""Sizes that the entry points accept and refuse, checked without a device (an accepted call then fails for want of one)."""
import ctypes

import numpy as np
import pytest

import paper_2301_08527_b200 as rk

EUNSUPPORTED, ECUDA = -3, -5


@pytest.fixture(scope="module", autouse=True)
def _no_device():
    import torch
    if torch.cuda.is_available():
        pytest.skip("passes addresses that are none")
    from paper_2301_08527_b200.build import build
    build()


def test_minirocket_batches_are_limited_by_features_only():
    lib = rk.load_library()
    m = rk.MiniRocket.create(3, 1, 50000, 9996)
    zeros = np.zeros(9996, np.float32)
    assert lib.rocket_mini_set_biases(m.handle, zeros.ctypes.data) == 0
    slices = int(sum((n + 7) // 8 for n in np.diff(m.host_arrays()["feature_offset"])))
    call = lambda n: lib.rocket_mini_transform(m.handle, ctypes.c_void_p(64), n, 1, 50000, ctypes.c_void_p(64), None)  # noqa: E731
    for n in (1, 150000, 200000, 0x7fffffff // slices):      # 200,000 univariate series of 50,000: 40 GB
        assert call(n) == ECUDA, n
    assert call(0x7fffffff // slices + 1) == EUNSUPPORTED
    m.close()
