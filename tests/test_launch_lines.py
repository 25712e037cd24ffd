"""Both sides of every line of the automatic launch shape (clusters of 8, 4 and
2 CTAs, one CTA of 512, 256 or 128 threads): the answers are those of one
explicitly shaped launch, and each side takes the shape it is meant to."""
import pytest

torch = pytest.importorskip("torch")

from paper_2201_13007_gb300 import synth  # noqa: E402

# (queries, L, M) and the automatic (CTAs per query, threads) on a GPU of 152 SMs
LINES = [
    ((12, 100, 8), (8, 256)), ((13, 100, 8), (4, 256)), ((33, 100, 8), (4, 256)), ((34, 100, 8), (2, 256)),
    ((76, 48, 4), (2, 128)), ((77, 48, 4), (1, 256)), ((304, 100, 8), (1, 512)), ((305, 100, 8), (1, 256)),
    ((608, 100, 8), (1, 256)), ((609, 100, 8), (1, 128)), ((609, 100, 32), (1, 256)), ((1300, 400, 8), (1, 128)),
    ((1000, 1024, 8), (1, 256)),
]


@pytest.mark.gpu
@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_every_launch_shape_gives_the_same_answers(storage):
    from paper_2201_13007_gb300.index import Index
    w = synth.make_workload("sift", 20000, 1300)
    ix = Index(w.base, w.adj, w.entry, storage=storage, keep_f32=storage != "f32")
    q = torch.from_numpy(w.queries).cuda()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for (nq, L, M), shape in LINES:
        d = ix.describe(nq, 10, L, M)
        if sms == 152:
            assert (d["cluster"], d["threads"]) == shape, (nq, L, M, d)
        for kw in ({}, {"rerank": True}, {"persistent": True}):
            got = ix.search(q[:nq], 10, L, M, **kw)
            ref = ix.search(q[:nq], 10, L, M, cluster=1, threads=128, hash_bits=14, rerank="rerank" in kw)
            assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1]), (nq, L, M, kw)
    ix.close()
