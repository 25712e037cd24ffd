"""The step's merge at the sizes where its forms meet: queues of one entry, of
a power of four and one more, survivors below, at and above the number that is
ranked instead of sorted, and visited sets so small that an id is met again
while it is queued, or twice in one step.

Every other base row equals the one before it, so that most keys are tied and
only the id orders them. Rows are integers in 0..255: results equal the
oracle's bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from parity_util import compare_exact  # noqa: E402
from paper_2201_13007_gb300 import synth  # noqa: E402




@pytest.fixture(scope="module")
def env():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2201_13007_gb300.index import Index
    w = synth.make_workload("sift", 20000, 24)
    base = w.base.copy()
    base[1::2] = base[::2]
    ix = Index(base, w.adj, w.entry)
    yield base, w, ix
    ix.close()


@pytest.mark.gpu
@pytest.mark.parametrize("L,M", [(1, 1), (4, 3), (33, 8), (64, 64), (129, 16), (257, 64), (1024, 64), (2048, 33)])
def test_merge_forms_agree_with_the_oracle(env, oracle_mod, L, M):
    base, w, ix = env
    k = min(L, 10)
    q = torch.from_numpy(w.queries).cuda()
    o_ids, o_keys, _ = oracle_mod.search(base, w.adj, w.entry, w.queries, algo="topm", L=L, K=k, M0=1, M_max=M, t=1,
                                         nthreads=8)
    for threads in (64, 128, 256, 512):
        for hash_bits, mode in ((8, 4), (8, 3), (12, 4)):
            ids, d = ix.search(q, k, L, M, threads=threads, hash_bits=hash_bits, visited_mode=mode, cluster=1)
            compare_exact(ids.cpu().numpy(), d.cpu().numpy(), o_ids, o_keys)
    for cluster, threads in ((2, 512), (8, 128)):
        ids, d = ix.search(q, k, L, M, threads=threads, hash_bits=8, cluster=cluster)
        compare_exact(ids.cpu().numpy(), d.cpu().numpy(), o_ids, o_keys)


def test_prefetch_lines_cover_a_row():
    """The lines asked of L2 are those a row touches, wherever it starts (the rule of prefetch_lines, restated)."""
    for row_bytes in range(16, 1025, 16):
        g = 128
        while row_bytes % g:
            g //= 2
        lines = (128 - g + row_bytes - 1) // 128 + 1
        for row in range(64):
            p = row * row_bytes
            touched = set(range(p // 128, (p + row_bytes - 1) // 128 + 1))
            asked = {(p + 128 * i) // 128 for i in range(lines - 1)} | {(p + row_bytes - 1) // 128}
            assert touched <= asked and len(asked - touched) == 0, (row_bytes, row)


@pytest.mark.gpu
@pytest.mark.parametrize("C", [2, 4, 8])
@pytest.mark.parametrize("hash_bits", [0, 8])
def test_one_cta_of_a_cluster_owns_every_vertex(oracle_mod, C, hash_bits):
    """Only ids that are multiples of 8 are reachable: one CTA finds every survivor, more than its share of the
    exchange buffers, in steps with few and with many of them."""
    from paper_2201_13007_gb300.index import Index
    g = np.random.Generator(np.random.PCG64(2))
    m, R, d = 3000, 32, 32
    n = 8 * m
    base = g.integers(0, 256, (n, d)).astype(np.float32)
    adj = np.full((n, R), -1, np.int32)
    adj[::8] = 8 * g.integers(0, m, (m, R))
    q = g.integers(0, 256, (6, d)).astype(np.float32)
    ix = Index(base, adj, 0)
    for L, M in ((40, 8), (300, 16), (600, 64)):
        o_ids, o_keys, _ = oracle_mod.search(base, adj, 0, q, algo="topm", L=L, K=10, M0=1, M_max=M, t=1, nthreads=8)
        ids, dists = ix.search(torch.from_numpy(q).cuda(), 10, L, M, cluster=C, hash_bits=hash_bits)
        compare_exact(ids.cpu().numpy(), dists.cpu().numpy(), o_ids, o_keys)
    ix.close()


@pytest.mark.gpu
@pytest.mark.parametrize("L,M", [(40, 32), (300, 16), (700, 64), (1500, 48)])
def test_wide_first_steps(env, oracle_mod, L, M):
    """M from the first step on: hundreds of survivors meet a queue of a few dozen, so that many fall between the same
    two entries, and a queue that overflows at once."""
    base, w, ix = env
    q = torch.from_numpy(w.queries).cuda()
    o_ids, o_keys, _ = oracle_mod.search(base, w.adj, w.entry, w.queries, algo="topm", L=L, K=10, M0=M, M_max=M, t=1,
                                         nthreads=8)
    for threads, cluster in ((64, 1), (128, 1), (256, 1), (512, 1), (256, 4)):
        for hash_bits in (8, 13):
            ids, d = ix.search(q, 10, L, M, M0=M, threads=threads, hash_bits=hash_bits, cluster=cluster, visited_mode=4)
            compare_exact(ids.cpu().numpy(), d.cpu().numpy(), o_ids, o_keys)
