"""How many kernels a planned batch launches on both sides of its line, 32
queries per SM, with and without a launch configuration."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2201_13007_gb300 import synth  # noqa: E402


def _kernels(batch, q):
    """Kernel nodes of one search captured into a CUDA graph."""
    out = batch.search(q)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        batch.search(q, out=out, stream=side)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        batch.search(q, out=out)
    cuda = ctypes.CDLL("libcuda.so.1")
    g, n = ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t()
    assert cuda.cuGraphGetNodes(g, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cuda.cuGraphGetNodes(g, nodes, ctypes.byref(n)) == 0
    kinds = []
    for node in nodes:
        kind = ctypes.c_int()
        assert cuda.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        kinds.append(kind.value)
    return kinds.count(0)  # CU_GRAPH_NODE_TYPE_KERNEL


@pytest.mark.gpu
def test_launches_of_a_batch():
    from paper_2201_13007_gb300.index import Batch, Index
    line = 32 * torch.cuda.get_device_properties(0).multi_processor_count
    w = synth.make_workload("sift", 20000, line + 1)
    ix = Index(w.base, w.adj, w.entry, storage="bf16")
    R = ix.info()["R"]
    light = 256 // R  # the most entries a step of a light query expands
    auto, tuned, threads = None, [(64, 0, 0), (256, 0, 12)], [(64, 128, 0), (256, 0, 0)]
    for nq, Ms, buckets, want in ((line, (light, light + 1), auto, 2), (line + 1, (light, light + 1), auto, 4),
                                  (line + 1, (1, light), auto, 2), (line + 1, (light + 1, 64), auto, 2),
                                  (line + 1, (light, light + 1), tuned, 4), (line + 1, (light, light + 1), threads, 3)):
        g = np.random.default_rng(nq)
        L = g.choice([60, 200], nq).astype(np.int32)
        M = g.choice(Ms, nq).astype(np.int32)
        b = Batch(ix, np.full(nq, 10, np.int32), L, M, buckets=buckets)
        q = torch.from_numpy(w.queries[:nq]).cuda()
        assert b.n_buckets == 2
        assert _kernels(b, q) == want, (nq, Ms, buckets)
        b.close()
    ix.close()
