"""The tuner's choice against the library's own, with batches whose times are
given: a launch configuration that is the fastest for a sample alone is kept
only where the whole batch is faster with it. No GPU: the batch and the events
are stand-ins with a clock of their own."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2201_13007_gb300 import autotune  # noqa: E402

NOW = [0.0]


class _Event:
    def __init__(self, enable_timing=False):
        self.t = 0.0

    def record(self):
        self.t = NOW[0]

    def synchronize(self):
        pass

    def elapsed_time(self, end):
        return end.t - self.t


class _Index:
    def info(self):
        return {"n": 1, "d": 4, "R": 32, "storage": "bf16", "metric": "l2"}


def _whole(cost, L, buckets):
    """Time of a batch: cost(bucket's L_max, config, queries of the whole batch) for every query of each bucket."""
    t, lo = 0.0, 0
    for hi, th, hb in buckets:
        t += int(((L > lo) & (L <= hi)).sum()) * cost(hi, (th, hb), L.size)
        lo = hi
    return t


def _tune(monkeypatch, cost, L, **kw):
    class _Batch:
        def __init__(self, index, k, L, M, *, buckets=None, **params):
            if any(th == 128 and hb == 14 for _, th, hb in buckets):
                raise RuntimeError("does not fit")
            self.t = _whole(cost, np.asarray(L), buckets)

        def search(self, queries, out=None):
            NOW[0] += self.t
            return None, None

        def close(self):
            pass

    monkeypatch.setattr(autotune, "Batch", _Batch)
    monkeypatch.setattr(torch.cuda, "Event", _Event)
    monkeypatch.setattr(torch.cuda, "synchronize", lambda *a: None)
    one = np.ones_like(L)
    return autotune.tune_buckets(_Index(), torch.zeros((L.size, 4)), one, L, 8 * one, **kw)


def test_never_slower_than_the_librarys_choice(monkeypatch):
    L = np.random.default_rng(1).choice([64, 500, 1000], 20000).astype(np.int32)

    def cost(hi, cfg, nq):  # (256, 13) beats the library's shape alone, but not its two launches of a large bucket
        if hi == 1024:
            return 2.0 if cfg == (0, 0) and nq > 4864 else 3.0 if cfg == (256, 13) else 4.0
        if hi == 512:  # a choice that is better in the batch as well
            return 1.0 if cfg == (512, 14) else 1.5
        return 1.0

    got = _tune(monkeypatch, cost, L)
    auto = [(hi, 0, 0) for hi in autotune.LADDER]
    assert [b[0] for b in got] == list(autotune.LADDER)
    assert _whole(cost, L, got) <= _whole(cost, L, auto)
    assert dict((b[0], b[1:]) for b in got)[512] == (512, 14)
    assert dict((b[0], b[1:]) for b in got)[1024] == (0, 0)


def test_choice_of_a_small_batch(monkeypatch, tmp_path):
    L = np.full(300, 100, np.int32)
    cost = lambda hi, cfg, nq: 1.0 if cfg == (128, 11) else 2.0
    cache = str(tmp_path / "c" / "tune.json")
    got = _tune(monkeypatch, cost, L, cache_path=cache)
    assert dict((b[0], b[1:]) for b in got)[128] == (128, 11)
    assert _tune(monkeypatch, lambda *a: 1.0, L, cache_path=cache) == got  # read back
