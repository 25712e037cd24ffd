"""The automatic visited set of a few queries with the longest queues and
widest steps: 2^14 sets on one side of its lines, 2^13 on the other, and the
same answers."""
import pytest

torch = pytest.importorskip("torch")

from paper_2201_13007_gb300 import synth  # noqa: E402


@pytest.mark.gpu
def test_sets_of_long_queues():
    from paper_2201_13007_gb300.index import Index
    w = synth.make_workload("sift", 20000, 40)
    q = torch.from_numpy(w.queries).cuda()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for storage, long_rows in (("f32", 14), ("bf16", 13)):
        ix = Index(w.base, w.adj, w.entry, storage=storage)
        R = ix.info()["R"]
        for nq, L, M, bits in ((33, 1537, 2048 // R, long_rows), (33, 1536, 2048 // R, 13), (33, 1537, 2048 // R - 1, 13),
                               (sms, 2048, 64, long_rows), (sms + 1, 2048, 64, 13)):
            d = ix.describe(nq, 10, L, M)
            assert (d["cluster"], d["hash_bits"]) == (1, bits), (storage, nq, L, M, d)
        for L, M in ((1537, 64), (2048, 64)):
            got = ix.search(q, 10, L, M)
            ref = ix.search(q, 10, L, M, hash_bits=13 if long_rows == 14 else 14)
            assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
        ix.close()
