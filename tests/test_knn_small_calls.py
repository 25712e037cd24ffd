"""Small k-NN calls on both sides of the lines below which the scan kernel
answers alone: the rule as it is stated, and the oracle's rows bit for bit."""
import ctypes

import pytest

from native_util import compile_and_load
from test_knn import _bf16, _integer_rows
from test_knn_filter import _check

SHIM = r"""
#include "knn.cuh"
extern "C" int scan_alone(int64_t n, int64_t nq) { return ann::knn_scan_is_faster(n, nq); }
"""
# (base rows, queries, whether the scan answers alone)
LINES = [(1, 1, 1), (128, 16, 1), (128, 17, 0), (129, 16, 0), (128, 640, 0), (128, 641, 1), (320, 641, 1), (320, 640, 0),
         (321, 641, 0), (320, 4, 1), (320, 5, 0),
         (321, 4, 0), (321, 100000, 0), (20000, 1, 0), (5, 100000, 1)]


def test_the_rule(tmp_path):
    shim = compile_and_load(SHIM, str(tmp_path))
    for n, nq, scan in LINES:
        assert shim.scan_alone(ctypes.c_int64(n), ctypes.c_int64(nq)) == scan, (n, nq)


@pytest.mark.gpu
@pytest.mark.parametrize("metric", ["l2", "ip"])
def test_both_sides_of_the_lines(metric):
    for n, nq, _ in LINES[:12]:
        base, bits = _bf16(_integer_rows(n, 64, 7 + n))
        q, qbits = _bf16(_integer_rows(nq, 64, 8))
        _check(base, q, bits, qbits, -1, metric, 64)
