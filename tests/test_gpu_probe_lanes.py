"""The lane groups of the probe kernel (batches of 2048 queries and more, of up
to eight terms a query on average) and the list of long queries that a warp
each answers behind them: batches around 2048 queries, means around eight
terms, queries of 32 and 33 terms and of hundreds, none of them and all of a
lane group's; from host memory, from device memory (where the device picks the
instance) and through plans sized for more, replayed with batches below and
above 2048.  Every ID list equals the oracle's."""
import numpy as np
import pytest

import synth
from tests.parity import assert_query_equal

pytestmark = pytest.mark.gpu

# row widths of every number of lanes a group has (1 .. 32), K large enough for the probe path
LAYOUTS = [(300, 30, 3, 2), (700, 64, 5, 1), (300, 120, 8, 3), (900, 250, 4, 4), (2000, 500, 8, 2), (900, 1000, 2, 2),
           (1500, 2000, 3, 1), (400, 4096, 8, 2)]


def _batch(rng, lists):
    off = np.zeros(len(lists) + 1, np.uint64)
    np.cumsum([len(x) for x in lists], out=off[1:])
    return synth.Collection("keys", np.concatenate(lists), off)


@pytest.fixture(scope="module", params=LAYOUTS, ids=lambda p: "K%d_B%d_R%d_eta%d" % p)
def pair(request):
    from oracle.oracle import Oracle
    from paper_1910_02611_gb300 import Rambo

    K, B, R, eta = request.param
    rng = np.random.default_rng(B)
    vocab = rng.integers(0, 1 << 63, 60, dtype=np.uint64)
    g, o = Rambo(K, B, R, 1 << 12, eta, 5), Oracle(K, B, R, 1 << 12, eta, 5)
    # every set holds the first terms, fewer the later ones
    sets = _batch(rng, [vocab[: int(rng.integers(8, vocab.size + 1))] for _ in range(K)])
    ids = np.arange(K, dtype=np.uint64)
    g.insert(ids, sets.data, sets.offsets, kind="keys")
    o.insert_keys_batch(ids, sets.data, sets.offsets)
    yield rng, vocab, g, o
    g.close()


def _terms(rng, vocab, n):
    """n terms that some sets hold together, now and then an absent one among them"""
    x = vocab[rng.integers(0, int(rng.integers(1, vocab.size)), n)]
    if rng.random() < 0.2:
        x[rng.integers(0, n)] = rng.integers(0, 1 << 63, dtype=np.uint64)
    return x


def _everywhere(g, o, q, plan_for=None):
    import torch

    from paper_1910_02611_gb300 import Plan

    ids, off = assert_query_equal(g, o, q)
    ids_d, off_d = g.query(torch.from_numpy(q.data.view(np.int64)).cuda(),
                           torch.from_numpy(q.offsets.view(np.int64)).cuda(), kind="keys")
    assert np.array_equal(off_d.cpu().numpy().view(np.uint64), off)
    assert np.array_equal(ids_d.cpu().numpy().view(np.uint32), ids)
    if plan_for:
        plan = Plan(g, "keys", plan_for, max(q.data.size, 3 * plan_for), max(1, ids.size))
        for n in (len(q), 2047, len(q)):
            part = q.subset(np.arange(min(n, len(q))))
            plan.launch_host(part.data, part.offsets)
            ids_p, off_p = plan.wait()
            assert np.array_equal(off_p, off[: len(part) + 1])
            assert np.array_equal(ids_p, ids[: int(off[len(part)])])
        plan.close()
    return ids


def test_batches_around_the_least_size(pair):
    rng, vocab, g, o = pair
    for n in (2047, 2048, 2049, 5000):
        q = _batch(rng, [_terms(rng, vocab, int(rng.integers(1, 6))) for _ in range(n)])
        ids = _everywhere(g, o, q, plan_for=6000 if n in (2048, 5000) else None)
        assert ids.size > n


def test_means_around_eight_terms(pair):
    rng, vocab, g, o = pair
    for extra in (-1, 0, 1):  # terms in all: eight a query, one more, one less
        lists = [_terms(rng, vocab, 8) for _ in range(2100)]
        lists[77] = _terms(rng, vocab, 8 + extra)
        _everywhere(g, o, _batch(rng, lists))


@pytest.mark.parametrize("long", [[], [32], [33], [31, 32, 33, 34], [200, 33, 1000, 32]])
def test_long_queries_in_a_batch_of_short_ones(pair, long):
    rng, vocab, g, o = pair
    n = 3000
    lists = [_terms(rng, vocab, int(rng.integers(1, 4))) for _ in range(n)]
    at = [0, n - 1, 31, 32, 1500, 2999 - 40][: len(long)]
    for t, m in zip(at, long):
        lists[t] = np.concatenate([vocab[:4], vocab[rng.integers(0, 8, m - 4)]])
    _everywhere(g, o, _batch(rng, lists), plan_for=4000)
    # every query of some warps
    if long:
        for t in range(640, 640 + 64):
            lists[t] = vocab[rng.integers(0, 8, 33 + t % 3)]
        _everywhere(g, o, _batch(rng, lists), plan_for=4000)


def test_sequences_by_lane_groups():
    from oracle.oracle import Oracle
    from paper_1910_02611_gb300 import Rambo
    import torch

    w = synth.make("genome", 0.01, m=1 << 16)
    g, o = Rambo(w.K, w.B, w.R, w.m, w.eta, w.seed), Oracle(w.K, w.B, w.R, w.m, w.eta, w.seed)
    g.insert(w.sets.ids, w.sets.data, w.sets.offsets, kind="seq")
    o.insert_seq_batch(w.sets.ids, w.sets.data, w.sets.offsets, 31)
    rng = np.random.default_rng(3)
    # windows of 1 to 6 k-mers of the sets' own sequences, three of 32, 33 and 400
    length = 31 + rng.integers(0, 6, 3000)
    length[[5, 6, 2999]] = [62, 63, 430]
    q = synth.substring_queries(rng, w.sets, length, max_subst=0.0)
    for k in (31, 31 | 0x100, 31 | 0x200):
        data = q.data.copy()
        if k & 0x200:
            data[q.offsets[5:7].astype(np.int64)] = ord("N")
        want = o.query_batch("seq", data, q.offsets, k=k)
        assert want[0].size
        ids, off = g.query(data, q.offsets, kind="seq", k=k)
        assert np.array_equal(off, want[1]) and np.array_equal(ids, want[0])
        ids, off = g.query(torch.from_numpy(data).cuda(), torch.from_numpy(q.offsets.view(np.int64)).cuda(), kind="seq", k=k)
        assert np.array_equal(off.cpu().numpy().view(np.uint64), want[1])
        assert np.array_equal(ids.cpu().numpy().view(np.uint32), want[0])
    g.close()
