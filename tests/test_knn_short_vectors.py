"""k-NN of vectors so short that their squared norms come near the smallest
normal FP32 number (2^-126) or fall below it: no neighbour may be lost.

Integer rows times a power of two down to 2^-74 have keys that are exact in
FP32 (multiples of 2^-148), so results equal the oracle's bit for bit. Unit
rows times 1e-19 are compared under the FP32 error bound of a key, which below
2^-126 is the spacing 2^-149 of the numbers there."""
import numpy as np
import pytest

from test_knn import _bf16, _gpu_knn, _integer_rows, _oracle_knn, _unit_rows


@pytest.mark.gpu
@pytest.mark.parametrize("metric", ["l2", "ip"])
@pytest.mark.parametrize("d", [32, 64, 128])
def test_scaled_integer_rows(d, metric):
    n, k, rows = 6000, 64, slice(1000, 1300)
    x = _integer_rows(n, d, 5)
    oi, ok = _oracle_knn(x, x[rows], 1000, metric, k)  # a power of two changes no order
    for s in (20, 56, 64, 70, 71, 72, 73, 74):
        _, bits = _bf16(x * np.float32(2.0 ** -s))
        gi, gd = _gpu_knn(bits, bits[rows], 1000, metric, k)
        assert np.array_equal(gi, oi), s
        assert np.array_equal(gd.astype(np.float64), ok * 2.0 ** (-2 * s)), s


@pytest.mark.gpu
@pytest.mark.parametrize("scale", [1e-15, 1e-17, 1e-19])
def test_scaled_unit_rows(scale):
    n, d, k, rows = 4000, 96, 32, slice(0, 200)
    base, bits = _bf16(_unit_rows(n, d, 11) * np.float32(scale))
    gi, gd = _gpu_knn(bits, bits[rows], 0, "l2", k)
    oi, ok = _oracle_knn(base, base[rows], 0, "l2", k, extra=1)
    # |q|^2 + |x|^2 - 2<q, x>: (d + 2) u (|q| + |x|)^2, and at most 3 d + 2 roundings to multiples of 2^-149
    tol = (d + 2) * 2.0 ** -24 * (2 * 1.01 * scale) ** 2 + (3 * d + 2) * 2.0 ** -149
    x = base.astype(np.float64)
    for r in range(gi.shape[0]):
        exact = ((x[gi[r]] - x[r]) ** 2).sum(1)
        assert np.unique(gi[r]).size == k and (gi[r] >= 0).all()
        assert np.all(np.abs(gd[r] - exact) <= tol), r
        assert np.all(np.abs(exact - ok[r, :k]) <= 2 * tol), r
        gap = np.diff(np.r_[-np.inf, ok[r]])  # a rank clear of both neighbours holds the oracle's id
        clear = (gap[:k] > 2 * tol) & (gap[1:] > 2 * tol)
        assert np.array_equal(gi[r][clear], oi[r, :k][clear]), r
