"""The wide probe kernel's hand-over and the wide set kernel: tables that fit
shared memory at once and ones that take several passes, more than eight
tables (two partition-row reads), row strides of 1, 2 and more words, ID
spaces around 256 and 8192 IDs (a warp's and a block's step), and batches
around 16 queries (a group).  Every ID list equals the oracle's."""
import numpy as np
import pytest

import synth
from tests.parity import assert_query_equal

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,B,R,eta", [
    (3073, 5000, 4, 2), (8193, 4200, 3, 3), (4096, 65535, 5, 1), (3000, 30, 9, 2), (3333, 60, 16, 4), (8192, 20001, 12, 1)])
def test_wide_set_kernel_at_tile_edges(K, B, R, eta):
    import torch

    from oracle.oracle import Oracle
    from paper_1910_02611_gb300 import Plan, Rambo

    rng = np.random.default_rng(K + B)
    vocab = rng.integers(0, 1 << 63, 200, dtype=np.uint64)
    pop = 1.0 / np.arange(1, vocab.size + 1)
    pop /= pop.sum()

    def collection(lists):
        off = np.zeros(len(lists) + 1, np.uint64)
        np.cumsum([len(x) for x in lists], out=off[1:])
        return synth.Collection("keys", np.concatenate(lists), off)

    ids = np.unique(np.concatenate([rng.choice(K, 1500, replace=False), [0, K - 1]])).astype(np.uint64)
    sets = collection([np.unique(rng.choice(vocab, int(rng.integers(1, 20)), p=pop)) for _ in ids])
    g, o = Rambo(K, B, R, 1 << 9, eta, 9), Oracle(K, B, R, 1 << 9, eta, 9)
    g.insert(ids, sets.data, sets.offsets, kind="keys")
    o.insert_keys_batch(ids, sets.data, sets.offsets)
    for n in (1, 15, 16, 17, 33, 200):
        q = collection([rng.choice(vocab, int(rng.integers(1, 7)), p=pop) for _ in range(n)])
        ids_h, off_h = assert_query_equal(g, o, q)
    ids_d, off_d = g.query(torch.from_numpy(q.data.view(np.int64)).cuda(),
                           torch.from_numpy(q.offsets.view(np.int64)).cuda(), kind="keys")
    assert np.array_equal(off_d.cpu().numpy().view(np.uint64), off_h)
    assert np.array_equal(ids_d.cpu().numpy().view(np.uint32), ids_h)
    plan = Plan(g, "keys", 300, q.data.size, max(1, ids_h.size))
    plan.launch_host(q.data, q.offsets)
    ids_p, off_p = plan.wait()
    assert np.array_equal(off_p, off_h) and np.array_equal(ids_p, ids_h)
    plan.close()
    g.close()
