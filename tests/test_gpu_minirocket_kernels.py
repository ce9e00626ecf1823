"""Both MINIROCKET kernels against the oracle, at shapes that test_minirocket_dispatch.py checks to be theirs: tiles of all channels
of a dilation, and one combination at a time (many channels, few tiles; whole rows and 256-column tiles, more than eight features)."""
import pytest

from test_gpu_minirocket import _check

# channels, steps, examples, features; one combination at a time
CASES = [(41, 5000, 2, 84 * 6, True), (64, 1500, 1, 84 * 10, True), (120, 9001, 2, 84 * 32, True), (20, 1501, 1, 84 * 10, True),
         (100, 64, 1, 84 * 120, True), (250, 700, 1, 84 * 5, True),
         (20, 700, 30, 84 * 12, False), (41, 500, 30, 84 * 12, False), (3, 333, 40, 84 * 30, False), (32, 1203, 12, 84 * 9, False)]


@pytest.mark.gpu
@pytest.mark.parametrize("C,L,N,F,walks", CASES)
def test_against_the_oracle(C, L, N, F, walks):
    _check(C, L, N, F, seed=700 + C, examples=[0, N - 1])
