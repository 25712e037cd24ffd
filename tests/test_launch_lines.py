"""Both sides of every line of the automatic launch shape (clusters of 8
CTAs, one CTA of 512, 256 or 128 threads): the answers are those of one
explicitly shaped launch, and each side takes the shape it is meant to."""
import pytest

torch = pytest.importorskip("torch")

from paper_2201_13007_gb300 import synth  # noqa: E402

# (queries, L, M) and the automatic (CTAs per query, threads) over 128-d FP32 and BF16 rows (512 and 256 bytes, 32 to a
# vertex) on a GPU of 152 SMs
LINES = [
    ((1, 48, 4), (1, 256), (1, 256)), ((8, 100, 11), (1, 256), (1, 256)), ((8, 100, 12), (8, 256), (1, 256)),
    ((8, 100, 64), (8, 512), (8, 512)), ((9, 100, 64), (1, 512), (1, 512)), ((152, 100, 32), (1, 512), (1, 512)),
    ((153, 100, 32), (1, 512), (1, 256)), ((304, 100, 24), (1, 512), (1, 256)), ((305, 100, 24), (1, 256), (1, 256)),
    ((608, 100, 8), (1, 256), (1, 256)), ((609, 100, 8), (1, 128), (1, 128)), ((609, 100, 32), (1, 256), (1, 256)),
    ((1000, 1024, 8), (1, 256), (1, 256)), ((1300, 400, 8), (1, 128), (1, 128)),
]


@pytest.mark.gpu
@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_every_launch_shape_gives_the_same_answers(storage):
    from paper_2201_13007_gb300.index import Index
    w = synth.make_workload("sift", 20000, 1300)
    ix = Index(w.base, w.adj, w.entry, storage=storage, keep_f32=storage != "f32")
    q = torch.from_numpy(w.queries).cuda()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for (nq, L, M), *shapes in LINES:
        shape = shapes[storage == "bf16"]
        d = ix.describe(nq, 10, L, M)
        if sms == 152:
            assert (d["cluster"], d["threads"]) == shape, (nq, L, M, d)
        for kw in ({}, {"rerank": True}, {"persistent": True}):
            got = ix.search(q[:nq], 10, L, M, **kw)
            ref = ix.search(q[:nq], 10, L, M, cluster=1, threads=128, hash_bits=14, rerank="rerank" in kw)
            assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1]), (nq, L, M, kw)
    ix.close()
