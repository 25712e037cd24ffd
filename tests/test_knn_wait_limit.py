"""A k-NN call whose waits run out: the filter kernel gives up, no later kernel
of the call reads the lists that were not written, and the error word comes
back. The loads are left out, so that every wait for data of the first launch
runs out, over a workspace full of bytes that would be no valid count or id."""
import ctypes
import time

import numpy as np
import pytest

from native_util import compile_and_load
from test_knn import _bf16, _gpu_knn, _integer_rows

SHIM = r"""
#include "knn.cuh"
extern "C" {
// [0] the workspace's bytes, [1] where its error word lies
void plan(int64_t n, int64_t nq, int sms, int64_t *out) {
    const ann::KnnPlan p = ann::knn_plan(n, nq, sms);
    out[0] = (int64_t)p.bytes, out[1] = (int64_t)p.err;
}
int run(void *ws, const void *base, int64_t n, int d, int k, int sms, int no_loads, int32_t *ids, float *dists) {
    ann::KnnPlan p = ann::knn_plan(n, n, sms);
    p.no_loads = no_loads;
    return (int)ann::launch_knn_bf16(p, ws, base, n, d, base, n, 0, ANN_METRIC_L2, k, ids, dists, sms, nullptr);
}
}
"""


@pytest.mark.gpu
@pytest.mark.parametrize("n,d", [(300, 32), (3000, 96)])
def test_waits_that_run_out_are_reported(tmp_path, n, d):
    import torch
    shim = compile_and_load(SHIM, str(tmp_path))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    out = (ctypes.c_int64 * 2)()
    shim.plan(ctypes.c_int64(n), ctypes.c_int64(n), sms, out)
    _, bits = _bf16(_integer_rows(n, d, 3))
    base = bits.cuda()
    ws = torch.full((out[0],), 0x7F, dtype=torch.uint8, device="cuda")
    ids = torch.full((n, 10), -7, dtype=torch.int32, device="cuda")
    dists = torch.zeros((n, 10), dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()

    def run(no_loads):
        t0 = time.perf_counter()
        e = shim.run(ctypes.c_void_p(ws.data_ptr()), ctypes.c_void_p(base.data_ptr()), ctypes.c_int64(n), d, 10, sms,
                     no_loads, ctypes.c_void_p(ids.data_ptr()), ctypes.c_void_p(dists.data_ptr()))
        torch.cuda.synchronize()
        return e, int(ws[out[1]:out[1] + 4].view(torch.int32).item()), time.perf_counter() - t0

    e, err, seconds = run(1)
    assert (e, err) == (0, 2) and seconds < 1.0, (e, err, seconds)
    assert ((ids == -7) | (ids == -1)).all()  # no id was taken from the lists
    assert run(0)[:2] == (0, 0)  # the same workspace and context go on
    gi, gd = _gpu_knn(bits, bits, 0, "l2", 10)
    assert np.array_equal(ids.cpu().numpy(), gi) and np.array_equal(dists.cpu().numpy(), gd)
