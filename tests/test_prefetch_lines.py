"""The library's own prefetch_lines (how many 128-byte lines of a row are asked
of L2) for every row size: the lines asked for, the last of them by the row's
last byte, are those the row touches wherever it starts."""
import ctypes

from native_util import compile_and_load

SHIM = r"""
#include "ann_internal.cuh"
extern "C" int lines(int row_bytes) { return ann::prefetch_lines(row_bytes); }
"""


def test_prefetch_lines_of_the_library(tmp_path):
    shim = compile_and_load(SHIM, str(tmp_path))
    for row_bytes in range(16, 4097, 16):
        lines = shim.lines(row_bytes)
        if row_bytes > 1024:
            assert lines == 0, row_bytes  # prefetched whole
            continue
        for row in range(64):
            p = row * row_bytes
            touched = set(range(p // 128, (p + row_bytes - 1) // 128 + 1))
            asked = {(p + 128 * i) // 128 for i in range(lines - 1)} | {(p + row_bytes - 1) // 128}
            assert asked == touched, (row_bytes, row)
