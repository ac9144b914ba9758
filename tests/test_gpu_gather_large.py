"""The gather where a bitmap has more words than eight parts of 2048, and 128
of 128: single answers, a few, and batches that fill the grid, dense and of one
ID.  The answers of each term equal the oracle's wherever it is asked."""
import numpy as np
import pytest

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
