"""The gather at the ends of its cut into parts: bitmaps of more words than
eight parts of 2048 hold, and 128 of the smallest, and bitmaps of one to four
of the smallest; single answers, a few, and batches that fill the grid, dense
and of one ID.  Every ID list equals the oracle's."""
import numpy as np
import pytest

import synth
from tests.parity import assert_query_equal

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [524_289, 1_300_000])
def test_answers_over_large_id_spaces(K):
    import torch

    from oracle.oracle import Oracle
    from paper_1910_02611_gb300 import Rambo

    rng = np.random.default_rng(K)
    g, o = Rambo(K, 600, 2, 1 << 10, 1, 4), Oracle(K, 600, 2, 1 << 10, 1, 4)
    terms = rng.integers(0, 1 << 63, 4, dtype=np.uint64)
    ids = np.arange(0, K, 2, dtype=np.uint64)
    # every second set holds the first term, those of the middle eighth the second, one set the third
    eighth = ids[(ids >= K // 2) & (ids < K // 2 + K // 8)]
    data = np.concatenate([np.full(ids.size, terms[0]), np.full(eighth.size, terms[1]), terms[2:3]])
    owner = np.concatenate([ids, eighth, ids[-1:]])
    order = np.argsort(owner, kind="stable")
    data, owner = data[order], owner[order]
    off = np.searchsorted(owner, np.append(ids, K)).astype(np.uint64)
    g.insert(ids, data, off, kind="keys")
    o.insert_keys_batch(ids, data, off)
    rids, roff = o.query_batch("keys", terms, np.arange(5, dtype=np.uint64))
    want = [torch.from_numpy(rids[int(a) : int(b)].view(np.int32)).cuda() for a, b in zip(roff[:-1], roff[1:])]
    assert want[0].numel() >= ids.size and want[2].numel() >= 1
    for n in (1, 2, 5, 57, 900):
        for pick in ([0], [2], [0, 1, 2, 3]):
            which = rng.choice(pick, n)
            q = torch.from_numpy(terms[which].view(np.int64)).cuda()
            got, ends = g.query(q, torch.arange(n + 1, device="cuda"), kind="keys")
            ends = ends.tolist()
            assert [b - a for a, b in zip(ends[:-1], ends[1:])] == [want[t].numel() for t in which]
            for i, t in enumerate(which):
                assert torch.equal(got[ends[i] : ends[i + 1]].view(torch.int32), want[t])
            del got
    g.close()


@pytest.mark.parametrize("K", [2049, 2500, 4000, 4097, 8191])
def test_a_few_answers_over_a_few_thousand_sets(K):
    """Parts of 64 words: bitmaps of one more than that, of just under and over two, and of four."""
    from oracle.oracle import Oracle
    from paper_1910_02611_gb300 import Rambo

    rng = np.random.default_rng(K)
    g, o = Rambo(K, 40, 3, 1 << 8, 2, 4), Oracle(K, 40, 3, 1 << 8, 2, 4)
    keys = rng.integers(0, 1 << 63, 3, dtype=np.uint64)
    # the first key in every set, the second in the last 900, the third in one
    lists = [keys[: 1 + (i >= K - 900)] for i in range(K)]
    lists[K - 2] = keys
    off = np.zeros(K + 1, np.uint64)
    np.cumsum([x.size for x in lists], out=off[1:])
    ids = np.arange(K, dtype=np.uint64)
    g.insert(ids, np.concatenate(lists), off, kind="keys")
    o.insert_keys_batch(ids, np.concatenate(lists), off)
    for n in (17, 64, 300, 3000):  # (fewer go to the query kernel)
        q = keys[rng.integers(0, 3, n)]
        assert_query_equal(g, o, synth.Collection("keys", q, np.arange(n + 1, dtype=np.uint64)))
    g.close()
