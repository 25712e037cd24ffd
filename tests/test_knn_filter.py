"""The tensor-core filter in front of the k-NN results: edges of its tiles
(128 query rows, 256 base rows), of its nested samples of the base (each twice
the last, from at most 256 rows), of the split of one block of queries over
several CTAs, and the blocks it hands to the scan kernel (equal distances that
overrun its lists, magnitudes its bounds do not cover).

Rows are integers in 0..255 (times a power of two), so keys are exact in FP32
in any order of summation and results equal the oracle's bit for bit.
"""
import numpy as np
import pytest

from test_knn import _bf16, _gpu_knn, _integer_rows, _oracle_knn

# (d, metric, n, queries, k): queries = ("self", lo, hi) rows of the base, or ("new", count)
CASES = [
    (32, "l2", 1, ("new", 1), 3),
    (32, "ip", 64, ("self", 0, 64), 64),
    (64, "l2", 255, ("new", 128), 64),
    (64, "l2", 256, ("self", 0, 256), 64),
    (64, "ip", 257, ("self", 128, 257), 64),
    (96, "l2", 511, ("new", 127), 1),
    (96, "l2", 513, ("self", 500, 513), 64),
    (128, "l2", 1025, ("self", 0, 1025), 64),
    (128, "ip", 20011, ("new", 3), 64),
    (96, "l2", 33333, ("self", 33000, 33333), 64),
]


def _check(base, q, bits, qbits, self_offset, metric, k):
    gi, gd = _gpu_knn(bits, qbits, self_offset, metric, k)
    oi, ok = _oracle_knn(base, q, self_offset, metric, k)
    assert np.array_equal(gi, oi)
    fin = np.isfinite(ok)
    assert np.array_equal(np.isfinite(gd), fin)
    assert np.array_equal(gd[fin].astype(np.float64), ok[fin])


@pytest.mark.gpu
@pytest.mark.parametrize("case", CASES, ids=[f"d{c[0]}-{c[1]}-n{c[2]}-{c[3][0]}{c[3][-1]}-k{c[4]}" for c in CASES])
def test_filter_edges(case):
    d, metric, n, qs, k = case
    base, bits = _bf16(_integer_rows(n, d, 7 + n))
    if qs[0] == "self":
        lo, hi = qs[1], qs[2]
        _check(base, base[lo:hi], bits, bits[lo:hi], lo, metric, k)
    else:
        q, qbits = _bf16(_integer_rows(qs[1], d, 8 + d))
        _check(base, q, bits, qbits, -1, metric, k)


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["sorted", "copies", "zeros", "large"])
def test_filter_hands_over(kind):
    """Bases that strain the samples or the lists: sorted by cluster; thousands of equal rows (every distance
    ties at the bound); all rows zero; values whose squares pass the range of the filter's bounds."""
    n, d = 6000, 64
    g = np.random.Generator(np.random.PCG64(3))
    x = _integer_rows(n, d, 5)
    scale = 1.0
    if kind == "sorted":
        x = x[np.lexsort(x.T[::-1])]
    elif kind == "copies":
        x[g.permutation(n)[:4000]] = x[17]
    elif kind == "zeros":
        x[:] = 0.0
    else:
        scale = 2.0 ** 40
    base, bits = _bf16(x * np.float32(scale))
    rows = slice(1000, 1200)
    gi, gd = _gpu_knn(bits, bits[rows], 1000, "l2", 64)
    oi, ok = _oracle_knn(x, x[rows], 1000, "l2", 64)  # a power of two changes no order
    assert np.array_equal(gi, oi)
    assert np.array_equal(gd.astype(np.float64), ok * scale * scale)


@pytest.mark.gpu
def test_not_finite_rows_return():
    """Rows that hold NaN or infinities: the call returns, and rows far from them are unaffected."""
    x = _integer_rows(1500, 32, 9)
    x[7, 3] = np.nan
    x[900, 0] = np.inf
    base, bits = _bf16(x)
    gi, gd = _gpu_knn(bits, bits[:300], 0, "l2", 8)
    assert gi.shape == (300, 8) and ((gi >= -1) & (gi < 1500)).all()


@pytest.mark.gpu
def test_without_room_for_the_lists():
    """With too little free device memory for the filter's lists (201 MB here) the scan kernel answers alone: the same
    bits."""
    import torch
    _, bits = _bf16(_integer_rows(3000, 32, 4))
    ref = _gpu_knn(bits, bits, 0, "l2", 20)
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    hold = torch.empty(free - (96 << 20), dtype=torch.uint8, device="cuda")
    try:
        got = _gpu_knn(bits, bits, 0, "l2", 20)
    finally:
        del hold
        torch.cuda.empty_cache()
    assert np.array_equal(ref[0], got[0]) and np.array_equal(ref[1], got[1])
