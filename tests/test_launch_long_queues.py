"""Few queries with long queues: the automatic launch shape on both sides of
its lines (clusters of 4 CTAs from L = 512 and 96 or 128 KB of rows a step), and the
answers of one explicitly shaped launch."""
import pytest

torch = pytest.importorskip("torch")

from paper_2201_13007_gb300 import synth  # noqa: E402

# (queries, L, M) and the automatic (CTAs per query, threads) over 128-d FP32 and BF16 rows (512 and 256 bytes, 32 to a
# vertex), for any GPU of at least 64 SMs
LINES = [
    ((8, 511, 8), (1, 256), (1, 256)), ((8, 512, 8), (4, 256), (1, 256)), ((8, 512, 6), (4, 256), (1, 256)),
    ((8, 512, 5), (1, 256), (1, 256)),
    ((1, 512, 11), (4, 256), (1, 256)), ((1, 512, 15), (8, 256), (1, 256)), ((1, 512, 16), (8, 256), (4, 256)),
    ((8, 2048, 11), (4, 256), (1, 256)), ((8, 2048, 23), (8, 256), (4, 256)), ((9, 2048, 11), (1, 256), (1, 256)),
]


@pytest.mark.gpu
@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_long_queues(storage):
    from paper_2201_13007_gb300.index import Index
    w = synth.make_workload("sift", 20000, 16)
    ix = Index(w.base, w.adj, w.entry, storage=storage, keep_f32=storage != "f32")
    q = torch.from_numpy(w.queries).cuda()
    for (nq, L, M), *shapes in LINES:
        d = ix.describe(nq, 10, L, M)
        assert (d["cluster"], d["threads"]) == shapes[storage == "bf16"], (nq, L, M, d)
        for kw in ({}, {"rerank": True}):
            got = ix.search(q[:nq], 10, L, M, **kw)
            ref = ix.search(q[:nq], 10, L, M, cluster=1, threads=128, hash_bits=14, **kw)
            assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1]), (nq, L, M, kw)
    ix.close()


@pytest.mark.gpu
def test_long_rows_stay_on_one_cta():
    """960-d FP8 rows (960 bytes) of 120 to 180 KB a step; 132-d FP32 rows (528 bytes)."""
    from paper_2201_13007_gb300.index import Index
    g = torch.Generator().manual_seed(1)
    for d, storage, M in ((960, "e4m3", 6), (132, "f32", 8)):
        base = torch.rand((2000, d), generator=g).numpy()
        adj = torch.randint(0, 2000, (2000, 32), generator=g).to(torch.int32).numpy()
        ix = Index(base, adj, 0, storage=storage)
        assert ix.describe(8, 10, 1024, M)["cluster"] == 1
        ix.close()
