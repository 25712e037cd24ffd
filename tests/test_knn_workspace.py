"""The device memory of a k-NN call: within what the header promises for any
size, and the scan alone, with the same bits, where it cannot be had."""
import ctypes

import numpy as np
import pytest

from native_util import compile_and_load
from test_knn import _bf16, _gpu_knn, _integer_rows

SHIM = r"""
#include "knn.cuh"
extern "C" int64_t plan_bytes(int64_t n, int64_t nq, int sms) { return (int64_t)ann::knn_plan(n, nq, sms).bytes; }
"""


def test_workspace_is_what_the_header_says(tmp_path):
    shim = compile_and_load(SHIM, str(tmp_path))
    shim.plan_bytes.restype = ctypes.c_int64
    sizes = [1, 64, 255, 256, 257, 511, 513, 1000, 1025, 5000, 20011, 200000, 1000003, 10000000, 2 ** 31 - 1]
    queries = sizes + [3000, 3650, 7296, 7424, 14592, 14720, 29184, 29312, 58240, 58368, 58369]
    for n in sizes:
        # each of the nested samples is padded to whole tiles
        base = 36 * n + (320 << 10)
        for nq in queries:
            got = shim.plan_bytes(ctypes.c_int64(n), ctypes.c_int64(nq), 152)
            rows = -(-min(nq, 58368) // 128) * 128
            shares = max(1, min(32, -(-n // 2048)))
            assert got <= base + min(302 * 10 ** 6, rows * (1100 + 2100 * shares)), (n, nq, got)


@pytest.mark.gpu
def test_no_room_for_the_lists_of_few_queries():
    import torch
    _, bits = _bf16(_integer_rows(20000, 32, 4))  # 206 MB of workspace for 3,000 queries
    q = bits[:3000]
    ref = _gpu_knn(bits, q, 0, "l2", 20)
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (96 << 20), dtype=torch.uint8, device="cuda")
    try:
        got = _gpu_knn(bits, q, 0, "l2", 20)
    finally:
        del hold
        torch.cuda.empty_cache()
    assert np.array_equal(ref[0], got[0]) and np.array_equal(ref[1], got[1])
