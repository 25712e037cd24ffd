"""The work this library is used for, as cases that can be timed and compared.

Three kinds of call:

- ``search``: ``Index.search`` (or ``Index.search_host`` with ``host`` set) of ``nq`` queries over an index
  that the program keeps;
- ``batch``: a planned ``Batch`` of queries with uneven k, L and M;
- ``knn``: ``graph.knn_bf16``, the exact neighbour lists a similarity graph is built from.

The asynchronous walkers are left out: their visited set is updated in no fixed order, so two runs on the
same inputs give different ids and cannot be compared.

Point sets are mixtures of low intrinsic dimension (the neighbour lists of isotropic data of these dimensions
have no structure to search): ``sift`` integers 0..255, ``deep`` unit vectors, ``gist`` positive log-normal
rows. The graph over them is the usual one, built by a quicker recipe than the package's own (the candidate
lists come from overlapping blocks of nearby points instead of all pairs): candidates, occlusion prune,
reverse edges, one long-range edge in a free slot, entry at the medoid.
"""
import math

import numpy as np
import torch

from paper_2201_13007_gb300 import graph
from paper_2201_13007_gb300.index import Batch, Index

STORED = {"f32": 4, "bf16": 2, "f16": 2, "e4m3": 1}


def _search(name, data, n, d, nq, k, L, M, **more):
    case = {"name": name, "kind": "search", "data": data, "n": n, "d": d, "R": 32, "nq": nq, "k": k, "L": L, "M": M,
            "storage": "f32", "metric": "ip" if data == "deep" else "l2", "rerank": False, "persistent": False,
            "host": False}
    case.update(more)
    return case


def listed():
    return [
        # an interactive lookup: one query at the recall-0.99 latency point
        _search("one_query", "sift", 1_000_000, 128, 1, 10, 576, 64),
        # a handful of lookups at the cheapest serving point, BF16 rows without a second FP32 copy
        _search("eight_queries", "deep", 1_000_000, 96, 8, 10, 100, 8, storage="bf16"),
        # a small program of odd shape: few points, a dimension and a queue that are no multiples of anything
        _search("odd_333", "deep", 30_011, 100, 333, 7, 75, 6, R=24, metric="l2"),
        # a server's group of requests, from host memory and back
        _search("host_256", "deep", 1_000_000, 96, 256, 10, 192, 16, storage="bf16", host=True),
        # offline batches at recall 0.9 and 0.99: BF16 rows, FP32 re-rank
        _search("batch_r90", "sift", 1_000_000, 128, 10_000, 10, 128, 32, storage="bf16", rerank=True, persistent=True),
        _search("batch_r99", "sift", 1_000_000, 128, 10_000, 10, 576, 32, storage="bf16", rerank=True, persistent=True),
        # the same in plain FP32, one launch of one block per query
        _search("batch_f32", "sift", 1_000_000, 128, 10_000, 10, 576, 32),
        # long rows in 16 and 8 bits: high recall and quick
        _search("gist_f16", "gist", 200_000, 960, 1_000, 10, 768, 16, storage="f16", rerank=True, persistent=True),
        _search("gist_e4m3", "gist", 200_000, 960, 1_000, 10, 128, 8, storage="e4m3", rerank=True, persistent=True),
        # a day's requests of all kinds, planned once
        {"name": "uneven_batch", "kind": "batch", "data": "deep", "n": 1_000_000, "d": 96, "R": 32, "nq": 20_000,
         "storage": "bf16", "metric": "ip"},
        # neighbour lists for a graph: a small integer set and a larger one of unit vectors
        {"name": "knn_20k", "kind": "knn", "data": "sift", "n": 20_000, "d": 128, "k": 64, "metric": "l2"},
        {"name": "knn_200k", "kind": "knn", "data": "deep", "n": 200_000, "d": 96, "k": 64, "metric": "l2"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    case = _draw(rng)
    while work(case)["bytes"] > 3e10:  # no more than the largest batch listed
        case["nq"] = case["nq"] * 2 // 3
    return case


def _draw(rng):
    kind = rng.choice(["search", "search", "search", "search", "batch", "knn"])
    if kind == "knn":
        return {"kind": "knn", "data": rng.choice(["deep", "sift"]), "n": _log(rng, 5_000, 200_000),
                "d": rng.choice([32, 64, 96, 128]), "k": rng.choice([10, 32, 64]), "metric": rng.choice(["l2", "l2", "ip"])}
    if kind == "batch":
        return {"kind": "batch", "data": rng.choice(["deep", "sift"]), "n": _log(rng, 100_000, 1_000_000),
                "d": rng.choice([96, 128, rng.randrange(32, 160)]), "R": rng.choice([24, 32]),
                "nq": _log(rng, 500, 20_000), "storage": rng.choice(["bf16", "f32"]), "metric": rng.choice(["ip", "l2"])}
    data = rng.choice(["sift", "sift", "deep", "deep", "gist"])
    storage = rng.choice(["f32", "bf16", "f16"]) if data != "gist" else rng.choice(["f32", "f16", "e4m3"])
    L = _log(rng, 32, 1024)
    nq = _log(rng, 1, 10_000 if data != "gist" else 1_000)
    persistent = nq > 8 and rng.random() < 0.6
    return {"kind": "search", "data": data,
            "n": _log(rng, 20_000, 1_000_000) if data != "gist" else _log(rng, 20_000, 200_000),
            "d": {"sift": rng.choice([128, 128, rng.randrange(24, 200)]),
                  "deep": rng.choice([96, 96, rng.randrange(24, 200)]),
                  "gist": rng.choice([960, 960, rng.randrange(200, 1000)])}[data],
            "R": rng.choice([32, 32, 24, 48]), "nq": nq, "k": min(L, rng.choice([1, 10, 10, 32, 100])), "L": L,
            "M": rng.choice([4, 8, 16, 32, 64, rng.randrange(1, 64)]), "storage": storage,
            "metric": rng.choice(["ip", "l2"]) if data == "deep" else "l2",
            "rerank": storage != "f32" and rng.random() < 0.6, "persistent": persistent,
            "host": rng.random() < 0.25}


# ------------------------------------------------------------------ inputs

def _points(data, d, counts, seed):
    """Point sets of the given sizes from one mixture, float32 on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda")

    r = min(d, 24)
    means = normal(96, r)
    A = normal(r, d) / math.sqrt(r)
    mu = normal(d) * 0.5 - 2.0
    out = []
    for count in counts:
        lab = torch.randint(0, 96, (count,), generator=g, device="cuda")
        y = (means[lab] + normal(count, r)) @ A
        if data == "sift":
            x = (128.0 + 40.0 * (y + 0.15 * normal(count, d))).round_().clamp_(0.0, 255.0)
        elif data == "gist":
            x = torch.exp(mu + 0.4 * y + 0.05 * normal(count, d))
        else:
            x = torch.nn.functional.normalize(y + 0.1 * normal(count, d), dim=1)
        out.append(x.contiguous())
    return out


def _graph(x, R, seed):
    """(adjacency int32 n x R, entry): every point goes with its two nearest of about n / 500 pivots, points are
    laid out pivot by pivot and cut into blocks, and each block's own nearest pairs are the candidates."""
    n = x.shape[0]
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    k, B = 24, min(1024, n)
    p = x[torch.randperm(n, generator=g, device="cuda")[:max(8, n // 500)]]
    p = p[torch.argsort(p @ torch.randn(x.shape[1], generator=g, device="cuda"))]
    near = torch.empty((n, 2), dtype=torch.int64, device="cuda")
    for a in range(0, n, 1 << 17):
        near[a:a + (1 << 17)] = ((p * p).sum(1) - 2.0 * (x[a:a + (1 << 17)] @ p.T)).topk(2, largest=False).indices
    cand = torch.empty((2, n, k), dtype=torch.int64, device="cuda")
    dist = torch.empty((2, n, k), dtype=torch.float32, device="cuda")
    for half in range(2):
        order = torch.argsort(near[:, half], stable=True)
        blocks = (n + B - 1) // B
        # the last block is filled up from the points before it: it ends with the last point
        start = (torch.arange(blocks, device="cuda") * B).clamp_(max=n - B)
        ids = order[start[:, None] + torch.arange(B, device="cuda")]
        step = max(1, (1 << 27) // (B * max(B, x.shape[1])))
        for a in range(0, blocks, step):
            v = x[ids[a:a + step]]
            s = (v * v).sum(-1)
            w = s[:, :, None] + s[:, None, :] - 2.0 * torch.bmm(v, v.transpose(1, 2))
            w.diagonal(dim1=1, dim2=2).fill_(float("inf"))
            w, i = w.topk(k, dim=2, largest=False)
            got = torch.gather(ids[a:a + step], 1, i.flatten(1)).view_as(i)
            # a point of the last two blocks may be in both: the later of them, one block at a time
            for b in ([slice(None)] if a + step < blocks else [slice(0, -1), slice(-1, None)]):
                to = ids[a:a + step][b].reshape(-1)
                cand[half, to] = got[b].reshape(-1, k)
                dist[half, to] = w[b].reshape(-1, k).clamp_(min=0.0)
    cand, dist = torch.cat([cand[0], cand[1]], 1), torch.cat([dist[0], dist[1]], 1)
    cand, o = cand.sort(dim=1, stable=True)
    dist = dist.gather(1, o)
    dist[:, 1:].masked_fill_(cand[:, 1:] == cand[:, :-1], float("inf"))
    dist, o = dist.sort(dim=1, stable=True)
    cand = cand.gather(1, o)
    adj = graph.occlusion_prune(x, cand, dist, R, batch=max(1 << 12, min(1 << 17, (1 << 30) // (48 * x.shape[1]))))
    del cand, dist, o
    adj = graph.reverse_fill(x, adj, R, chunk=max(1 << 16, (1 << 29) // x.shape[1]))
    # one long-range edge in the first free slot, where there is one
    far = torch.randint(0, n, (n,), generator=g, device="cuda").to(torch.int32)
    deg = (adj >= 0).sum(1)
    row = torch.nonzero(deg < R).flatten()
    adj[row, deg[row]] = far[row]
    return adj, graph.medoid(x)


def _mix(case, seed):
    """k, L, M of a planned batch, one of each per request."""
    g = np.random.Generator(np.random.PCG64(seed))
    nq = case["nq"]
    k = g.choice([1, 10, 100], nq)
    L = np.maximum(k, g.choice([32, 64, 128, 256, 512, 1024], nq))
    M = g.choice([4, 8, 16, 32], nq)
    return k.astype(np.int32), L.astype(np.int32), M.astype(np.int32)


def prepare(case, seed):
    if case["kind"] == "knn":
        return {"case": case, "rows": _points(case["data"], case["d"], [case["n"]], seed)[0].to(torch.bfloat16)}
    base, q = _points(case["data"], case["d"], [case["n"], case["nq"]], seed)
    adj, entry = _graph(base, case["R"], seed)
    state = {"case": case, "index": Index(base, adj, entry, storage=case["storage"], metric=case["metric"],
                                          keep_f32=case.get("rerank", False))}
    del base, adj
    torch.cuda.empty_cache()
    if case["kind"] == "batch":
        state["plan"] = Batch(state["index"], *_mix(case, seed))
    if case.get("host"):
        q = q.cpu().pin_memory()
        state["out"] = (torch.empty((case["nq"], case["k"]), dtype=torch.int64).pin_memory(),
                        torch.empty((case["nq"], case["k"]), dtype=torch.float32).pin_memory())
    state["q"] = q
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "knn":
        return graph.knn_bf16(state["rows"], case["k"], case["metric"])
    if case["kind"] == "batch":
        return state["plan"].search(state["q"])
    if case["host"]:
        return state["index"].search_host(state["q"], case["k"], case["L"], case["M"], out=state["out"],
                                          rerank=case["rerank"], persistent=case["persistent"])
    return state["index"].search(state["q"], case["k"], case["L"], case["M"], rerank=case["rerank"],
                                 persistent=case["persistent"])


def work(case):
    d, n = case["d"], case["n"]
    if case["kind"] == "knn":
        return {"bytes": n * d * 2 + n * case["k"] * 8, "flops": 2.0 * n * n * d}
    stored = d * STORED[case["storage"]] + (4 if case["storage"] == "e4m3" else 0)
    if case["kind"] == "batch":
        # the mean of L over the mix, and of k
        k, L, nq = 37.0, 353.0, case["nq"]
    else:
        k, L, nq = case["k"], case["L"], case["nq"]
    # every entry of the final queue is expanded (its adjacency row is read), and of the neighbours named there
    # about R / 3 a vertex are new and have their row read once
    rows = min(float(n), L * case["R"] / 3.0)
    moved = L * case["R"] * 4 + rows * stored + (L * d * 4 if case.get("rerank") else 0) + d * 4 + k * 12
    return {"bytes": nq * moved, "flops": nq * rows * d * (3 if case["metric"] == "l2" else 2)}


# ------------------------------------------------------------------- exact

def _stored64(x, storage):
    """The rows as the index holds them, in 64 bits."""
    if storage == "bf16":
        return x.to(torch.bfloat16).double()
    if storage == "f16":
        return x.to(torch.float16).double()
    if storage == "e4m3":
        s = x.abs().amax(1, keepdim=True) / 448.0
        s = torch.where(s > 0, s, torch.ones_like(s))
        return ((x / s).to(torch.float8_e4m3fn).float() * s).double()
    return x.double()


def _keys(rows, ids, q, l2):
    """Keys (nq x m) of the rows ids (nq x m) for the queries, in 64 bits."""
    out = torch.empty(ids.shape, dtype=torch.float64, device=ids.device)
    step = max(1, (1 << 26) // (ids.shape[1] * rows.shape[1]))
    for a in range(0, ids.shape[0], step):
        v = rows[ids[a:a + step]]
        if l2:
            out[a:a + step] = (v - q[a:a + step, None, :]).square_().sum(-1)
        else:
            out[a:a + step] = -torch.bmm(v, q[a:a + step, :, None])[..., 0]
    return out


def _by_key_then_id(key, ids):
    o = torch.argsort(ids, dim=1, stable=True)
    key, ids = key.gather(1, o), ids.gather(1, o)
    o2 = torch.argsort(key, dim=1, stable=True)
    return key.gather(1, o2), ids.gather(1, o2), o.gather(1, o2)


def _best_first(rows, full, adj, entry, q, k, L, M, l2):
    """Best-first search: keys of the k nearest found, ascending. The queue holds the L smallest (key, id) seen;
    each step expands its first m unchecked entries, m doubling from 1 to M."""
    n, inf = rows.shape[0], float("inf")
    nq = q.shape[0]
    ids = torch.full((nq, L), n, dtype=torch.int64, device=q.device)  # n: an empty place
    key = torch.full((nq, L), inf, dtype=torch.float64, device=q.device)
    done = torch.ones((nq, L), dtype=torch.bool, device=q.device)
    ids[:, 0], done[:, 0] = entry, False
    key[:, 0] = _keys(rows, ids[:, :1], q, l2)[:, 0]
    live, m = torch.arange(nq, device=q.device), 1
    while True:
        live = live[(~done[live]).any(1)]
        if not live.numel():
            break
        i0, k0, d0 = ids[live], key[live], done[live]
        take = (~d0) & ((~d0).cumsum(1) <= m)
        d0 |= take
        # the entries taken, padded to m with an empty one
        at = torch.where(take, torch.arange(L, device=q.device), L).sort(dim=1).values[:, :m]
        v = torch.cat([i0, torch.full_like(i0[:, :1], n)], 1).gather(1, at)
        u = torch.cat([adj, torch.full_like(adj[:1], -1)])[v].flatten(1).long()
        u = torch.where(u < 0, n, u).sort(dim=1).values
        u[:, 1:][u[:, 1:] == u[:, :-1]] = n
        known = i0.sort(dim=1).values
        pos = torch.searchsorted(known, u).clamp_(max=L - 1)
        u[known.gather(1, pos) == u] = n
        w = _keys(rows, u.clamp(max=n - 1), q[live], l2)
        w[u == n] = inf
        k1, i1, o = _by_key_then_id(torch.cat([k0, w], 1), torch.cat([i0, u], 1))
        d1 = torch.cat([d0, u == n], 1).gather(1, o)
        ids[live], key[live], done[live] = i1[:, :L], k1[:, :L], d1[:, :L]
        m = min(2 * m, M)
    if full is not None:
        key = _keys(full, ids.clamp(max=n - 1), q, l2).masked_fill_(ids == n, inf)
        key = _by_key_then_id(key, ids)[0]
    return key[:, :k]


def exact(case, seed):
    l2 = case["metric"] == "l2"
    if case["kind"] == "knn":
        x = prepare(case, seed)["rows"].double()
        s = (x * x).sum(1)
        out = torch.empty((case["n"], case["k"]), dtype=torch.float64, device="cuda")
        step = max(1, (1 << 29) // case["n"])
        for a in range(0, case["n"], step):
            b = min(case["n"], a + step)
            w = x[a:b] @ x.T
            w = s[a:b, None] + s - 2.0 * w if l2 else -w
            r = torch.arange(a, b, device="cuda")
            w[r - a, r] = float("inf")
            out[a:b] = w.topk(case["k"], dim=1, largest=False, sorted=True).values
        return [None, out]
    if case["kind"] == "batch" or case["nq"] * case["L"] * case["R"] * case["d"] > 1 << 35:
        return None
    if -(-case["nq"] // 500) * (case["L"] / case["M"] + 10) > 1500:
        return None
    base, q = _points(case["data"], case["d"], [case["n"], case["nq"]], seed)
    adj, entry = _graph(base, case["R"], seed)
    rows = _stored64(base, case["storage"])
    full = base.double() if case["rerank"] else None
    parts = [_best_first(rows, full, adj, entry, q[a:a + 500].double(), case["k"], case["L"], case["M"], l2)
             for a in range(0, case["nq"], 500)]
    return [None, torch.cat(parts)]
