"""Query rows that the k-NN filter cannot bound (norms far above the
distances: a common offset) pass no further value, and the scan's rows are
those of the oracle. Rows are integers: keys are exact."""
import ctypes

import numpy as np
import pytest

from native_util import compile_and_load
from test_knn import _bf16, _integer_rows, _oracle_knn

SHIM = r"""
#include "knn.cuh"
extern "C" {
// [0] the workspace's bytes, [1], [2] where its counts of values that passed lie, and how many bytes of them
void plan(int64_t n, int64_t nq, int sms, int64_t *out) {
    const ann::KnnPlan p = ann::knn_plan(n, nq, sms);
    out[0] = (int64_t)p.bytes, out[1] = (int64_t)p.counts, out[2] = (int64_t)p.chunk_blocks * 128 * 4 * p.splits * 4;
}
int run(void *ws, const void *base, int64_t n, int d, int k, int sms, int32_t *ids, float *dists) {
    const ann::KnnPlan p = ann::knn_plan(n, n, sms);
    return (int)ann::launch_knn_bf16(p, ws, base, n, d, base, n, 0, ANN_METRIC_L2, k, ids, dists, sms, nullptr);
}
}
"""


@pytest.mark.gpu
@pytest.mark.parametrize("offset,bounded", [(0, 5000), (192, 0), ("half", 2560)])
def test_rows_given_up_pass_nothing(tmp_path, offset, bounded):
    import torch
    shim = compile_and_load(SHIM, str(tmp_path))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n, d, k = 5000, 32, 20
    g = np.random.Generator(np.random.PCG64(5))
    if offset == "half":  # 2,560 rows (20 blocks) by themselves, then rows all within a few units of one another
        x = _integer_rows(n, d, 5)
        x[2560:] = 192 + g.integers(0, 2, (n - 2560, d))
    elif offset:
        x = (offset + g.integers(0, 2, (n, d))).astype(np.float32)
    else:
        x = _integer_rows(n, d, 5)
    base, bits = _bf16(x)
    o = (ctypes.c_int64 * 3)()
    shim.plan(ctypes.c_int64(n), ctypes.c_int64(n), sms, o)
    ws = torch.zeros(o[0], dtype=torch.uint8, device="cuda")
    b = bits.cuda()
    ids = torch.empty((n, k), dtype=torch.int32, device="cuda")
    dists = torch.empty((n, k), dtype=torch.float32, device="cuda")
    for _ in range(2):  # the flags of one call are not the next one's
        e = shim.run(ctypes.c_void_p(ws.data_ptr()), ctypes.c_void_p(b.data_ptr()), ctypes.c_int64(n), d, k, sms,
                     ctypes.c_void_p(ids.data_ptr()), ctypes.c_void_p(dists.data_ptr()))
        torch.cuda.synchronize()
        assert e == 0
        oi, ok = _oracle_knn(base, base, 0, "l2", k)
        assert np.array_equal(ids.cpu().numpy(), oi) and np.array_equal(dists.cpu().numpy().astype(np.float64), ok)
    passed = ws[o[1]:o[1] + o[2]].view(torch.int32).view(-1, o[2] // (4 * 5120)).sum(1).cpu().numpy()  # by row, last pass
    assert passed[:bounded].astype(bool).mean() > 0.99 if bounded else True
    assert (passed[bounded:] == 0).all()
