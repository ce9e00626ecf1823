"""Ridge fits whose Gram matrix is summed in integers (rocket_gram.cu), at the edges of its tiles, stages and slices.

From N N P = 3e8 on (smaller fits, among them the first nine here, take the FP64 kernel).  Rows around multiples of 64 and 128, columns around multiples of 64 and of a quadruple, more columns than a 32-bit sum takes at once, rows of
very different magnitude.  Against the dual system in float64.  What the weights may be off by: their rounding to FP32 (2^-24 each) plus
the errors of the two solutions, each of the order of 2^-53 times the condition number of the system.

Features one column or value of which is far larger than the others, against the dual system in 80 bits: the weights may be off by their
rounding and twice what the same system summed and solved in float64 is off by (another order of its sums changes that by less).
"""
import numpy as np
import pytest

import paper_2301_08527_b200 as rk

pytestmark = pytest.mark.gpu


def _fit(F, y, alpha):
    import torch
    w, b = rk.rocket_ridge_fit(torch.from_numpy(F).cuda(), torch.from_numpy(y).cuda(), alpha)
    return w.cpu().numpy().astype(np.float64), float(b)


def _dual(F, y, alpha):
    F, y = F.astype(np.float64), y.astype(np.float64)
    mu, ym = F.mean(0), y.mean()
    Fc = F - mu
    w = Fc.T @ np.linalg.solve(Fc @ Fc.T + alpha * np.eye(len(y)), y - ym)
    largest = np.linalg.norm(Fc, 2) ** 2
    return w, ym - mu @ w, 2.0 ** -24 + 4 * 2.0 ** -53 * (largest + alpha) / alpha


@pytest.mark.parametrize("N,P,kind", [(127, 7500, "shares"), (128, 7601, "shares"), (129, 7702, "shares"), (191, 3403, "shares"), (193, 40001, "shares"),
                                      (257, 2049, "shares"), (257, 2111, "scales"), (320, 1985, "shifted"), (641, 320, "shares"),
                                      (127, 18700, "shares"), (128, 18353, "shares"), (129, 18070, "shares"), (191, 8331, "shares"), (257, 4609, "shares"),
                                      (257, 4607, "scales"), (320, 2945, "shifted"), (641, 768, "shares")])
def test_fits_match_the_dual_system_in_float64(N, P, kind):
    rng = np.random.default_rng(N + P)
    F = rng.random((N, P))
    F[:, 1::2] = 2.0 + 0.7 * rng.normal(size=(N, P // 2))
    if kind == "scales":                                     # rows of very different magnitude, one of them constant
        F *= 10.0 ** rng.uniform(-3, 3, size=(N, 1))
        F[7] = 0.25
    if kind == "shifted":                                    # far from zero: the centred values have few bits of the samples' left
        F += 1000.0
    F = F.astype(np.float32)
    y = (F[:, :50].astype(np.float64) @ rng.normal(size=50) / 50 + rng.normal(size=N)).astype(np.float32)
    w, b = _fit(F, y, 1.0)
    rw, rb, bound = _dual(F, y, 1.0)
    assert np.linalg.norm(w - rw) <= bound * np.linalg.norm(rw)
    # the intercept is made from the stored weights
    assert abs(b - rb) <= (bound + 2.0 ** -23) * (np.linalg.norm(rw) * np.linalg.norm(F.astype(np.float64).mean(0)) + abs(rb))
    again, _ = _fit(F, y, 1.0)
    assert np.array_equal(w, again)


@pytest.mark.parametrize("N,P", [(897, 19003), (2305, 17001)])
def test_digits_of_several_chunks_of_columns(N, P):
    # two and three chunks, the last one shorter; the dual system on the device
    import torch
    rng = np.random.default_rng(N)
    F = rng.random((N, P), dtype=np.float32)
    F[:, 1::2] = 2.0 + 0.7 * rng.normal(size=(N, P // 2)).astype(np.float32)
    y = rng.normal(size=N).astype(np.float32)
    w, _ = _fit(F, y, 1.0)
    Fc, yc = torch.from_numpy(F).cuda().double(), torch.from_numpy(y).cuda().double()
    Fc, yc = Fc - Fc.mean(0), yc - yc.mean()
    G = Fc @ Fc.T
    rw = (Fc.T @ torch.linalg.solve(G + torch.eye(N, dtype=torch.float64, device="cuda"), yc)).cpu().numpy()
    bound = 2.0 ** -24 + 4 * 2.0 ** -53 * (float(G.trace()) + 1.0)   # the trace is more than the largest eigenvalue
    assert np.linalg.norm(w - rw) <= bound * np.linalg.norm(rw)


@pytest.mark.parametrize("N,P,launches", [(33, 500, 4), (200, 7499, 4), (200, 7500, 6), (64, 120000, 4), (897, 19003, 8)])
def test_every_kernel_of_a_fit_is_counted_once(N, P, launches):
    # means, Gram matrix, factorisation and weights; integers: the scales, and digits and their products per chunk
    import torch
    F, y = torch.rand((N, P), device="cuda"), torch.rand(N, device="cuda")
    before = rk.kernel_launch_count()
    rk.rocket_ridge_fit(F, y, 1.0)
    assert rk.kernel_launch_count() - before == launches


def _weights_in_80_bits(F, y, alpha):
    Fc = F.astype(np.longdouble)
    Fc -= Fc.mean(0)
    x = y.astype(np.longdouble)
    x -= x.mean()
    A = Fc @ Fc.T + np.longdouble(alpha) * np.eye(len(y), dtype=np.longdouble)
    for j in range(len(y)):                                  # L D L^T
        A[j + 1:, j] /= A[j, j]
        A[j + 1:, j + 1:] -= np.outer(A[j + 1:, j] * A[j, j], A[j + 1:, j])
        x[j + 1:] -= A[j + 1:, j] * x[j]
    x /= np.diag(A)
    for j in range(len(y) - 1, -1, -1):
        x[j] -= A[j + 1:, j] @ x[j + 1:]
    return Fc.T @ x


def _weights_in_64_bits(F, y, alpha):
    Fc, yc = F.astype(np.float64), y.astype(np.float64)
    Fc, yc = Fc - Fc.mean(0), yc - yc.mean()
    G = alpha * np.eye(len(y))
    for p in range(0, F.shape[1], 128):
        G += Fc[:, p:p + 128] @ Fc[:, p:p + 128].T
    return Fc.T @ np.linalg.solve(G, yc)


def _no_further_off_than_64_bits(F, y, alpha):
    w, _ = _fit(F, y, alpha)
    exact = _weights_in_80_bits(F, y, alpha)
    size = np.linalg.norm(exact)
    err, err64 = (float(np.linalg.norm(v - exact) / size) for v in (w, _weights_in_64_bits(F, y, alpha)))
    assert err <= 2.0 ** -24 + 2.0 * err64, (err, err64)


@pytest.mark.parametrize("kind,size,alpha", [("column", 1e5, 1e-3), ("column", 1e6, 1e-3), ("column", 1e6, 1.0), ("column", 1e7, 1.0), ("value", 1e7, 1.0), ("value", 1e8, 1.0)])
def test_one_large_column_or_value(kind, size, alpha):
    N, P = 160, 12001
    rng = np.random.default_rng(int(np.log10(size)))
    F = rng.random((N, P))
    F[:, 1::2] = 2.0 + 0.7 * rng.normal(size=(N, P // 2))
    y = (F[:, :50] @ rng.normal(size=50) / 50 + rng.normal(size=N)).astype(np.float32)
    if kind == "column":
        F[:, 1] *= size
    else:
        F[3, 5] = size
    _no_further_off_than_64_bits(F.astype(np.float32), y, alpha)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_values_that_are_not_finite_are_refused(bad):
    F = np.random.default_rng(1).random((200, 8000)).astype(np.float32)
    F[13, 77] = bad
    with pytest.raises(rk.RocketError) as refused:
        _fit(F, F[:, 0].copy(), 1.0)
    assert refused.value.status == -1                        # invalid argument
