"""A planned batch whose buckets run as two launches (queries of up to 256
slots a step, and the others): every row is that of its own search, on both
sides of the lines that decide it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2201_13007_gb300 import synth  # noqa: E402


@pytest.mark.gpu
@pytest.mark.parametrize("nq,Ms", [(4864, (8, 9)), (4865, (8, 9)), (5000, (1, 8)), (5000, (9, 64)), (5000, (3, 8, 24))])
def test_parts_give_the_rows_of_single_searches(nq, Ms):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2201_13007_gb300.index import Batch, Index
    w = synth.make_workload("sift", 20000, 5000)  # integer values: sums are exact
    ix = Index(w.base, w.adj, w.entry, storage="bf16", keep_f32=True)
    q = torch.from_numpy(w.queries[:nq]).cuda()
    g = np.random.default_rng(nq)
    k = g.choice([1, 10], nq).astype(np.int32)
    L = g.choice([33, 64, 200], nq).astype(np.int32)
    M = g.choice(Ms, nq).astype(np.int32)
    b = Batch(ix, k, L, M)
    assert b.n_buckets == 2
    ids, dists = b.search(q)
    for _ in range(2):  # the launches' work counters are reset by each call
        again = b.search(q)
    for kk, ll, mm in {(int(x), int(y), int(z)) for x, y, z in zip(k, L, M)}:
        rows = torch.from_numpy(np.flatnonzero((k == kk) & (L == ll) & (M == mm))).cuda()
        one = ix.search(q[rows], kk, ll, mm)
        assert torch.equal(ids[rows, :kk], one[0]) and torch.equal(dists[rows, :kk], one[1])
        assert (ids[rows, kk:] == -1).all()
    assert torch.equal(ids, again[0]) and torch.equal(dists, again[1])
    b.close()
    ix.close()
