"""Long queries shared by the warps of a block, on rows of one word (whose
other probe instances run in narrower blocks than the grouped one): single
queries, a few, and as many as leave a query two warps or one; from host
memory, from device memory and through plans; with the number of warps left
open and asked for.  Every ID list equals the oracle's."""
import numpy as np
import pytest

import synth
from tests.parity import assert_query_equal

pytestmark = pytest.mark.gpu


def _index(K, B, R, eta, cls):
    rng = np.random.default_rng(7)
    data = synth.random_bases(rng, K * 3000)
    off = (np.arange(K + 1) * 3000).astype(np.uint64)
    g = cls(K, B, R, 1 << 16, eta, 1)
    if hasattr(g, "insert"):
        g.insert(np.arange(K, dtype=np.uint64), data, off, kind="seq")
    else:
        g.insert_seq_batch(np.arange(K, dtype=np.uint64), data, off, 31)
    return g, data


def _queries(rng, data, K, n, length):
    at = rng.integers(0, K, n)
    return np.concatenate([data[3000 * i : 3000 * i + length] for i in at]), (np.arange(n + 1) * length).astype(np.uint64)


@pytest.mark.parametrize("B,R,eta", [(20, 3, 1), (32, 4, 2), (32, 8, 2), (31, 2, 4)])
def test_long_queries_on_rows_of_one_word(B, R, eta):
    import torch

    from oracle.oracle import Oracle
    from paper_1910_02611_gb300 import Plan, Rambo

    K, rng = 1100, np.random.default_rng(B + R)
    g, data = _index(K, B, R, eta, Rambo)
    o, _ = _index(K, B, R, eta, Oracle)
    base = g.get_config()
    for n, length in ((1, 3000), (3, 700), (40, 330), (1216, 45), (1217, 45), (1521, 45), (2000, 45)):
        q, off = _queries(rng, data, K, n, length)
        want = o.query_batch("seq", q, off, k=31)
        assert want[0].size >= n
        for wpq, wpb in ((0, 0), (2, 0), (8, 0), (8, 4), (4, 2), (1, 0)):
            if wpq and n > 1300:
                continue
            g.set_config(**{**base, "warps_per_query": wpq, "warps_per_block": wpb})
            ids, ends = assert_query_equal(g, o, synth.Collection("seq", q, off))
            ids, ends = g.query(torch.from_numpy(q).cuda(), torch.from_numpy(off.view(np.int64)).cuda(), kind="seq")
            assert np.array_equal(ends.cpu().numpy().view(np.uint64), want[1])
            assert np.array_equal(ids.cpu().numpy().view(np.uint32), want[0])
            plan = Plan(g, "seq", 1600 if n < 1600 else n, max(q.size, 1 << 16), want[0].size + 8)
            for _ in range(2):
                plan.launch_host(q, off)
                ids, ends = plan.wait()
                assert np.array_equal(ends, want[1]) and np.array_equal(ids, want[0])
            plan.close()
    g.close()


def test_rows_of_one_word_get_as_many_warps_a_query_as_wider_ones():
    """One query of 19970 k-mers, on rows of one word and of two."""
    from paper_1910_02611_gb300 import Plan, Rambo

    rng, best = np.random.default_rng(2), {}
    data, off = synth.random_bases(rng, 100 * 20_000), (np.arange(101) * 20_000).astype(np.uint64)
    for B in (32, 64):
        g = Rambo(100, B, 4, 1 << 20, 2, 1)
        g.insert(np.arange(100, dtype=np.uint64), data, off, kind="seq")
        q = data[40_000:60_000].copy()
        plan = Plan(g, "seq", 2, q.size, 4000)
        times = []
        for _ in range(40):
            plan.launch_host(q, np.array([0, q.size], np.uint64))
            ids, _ = plan.wait()
            times.append(plan.last_stats()["query_kernel_ms"])
        assert 2 in ids
        best[B] = min(times)
        plan.close()
        g.close()
    assert best[32] < 1.25 * best[64], best
