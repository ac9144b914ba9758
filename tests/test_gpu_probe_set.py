"""The probe path (lane groups, warps and warp groups) and the set kernel
behind it, at the edges of their tiles: ID spaces around 256 IDs (a warp's
step) and 2048 (a block's), batches around 32, 64 and 128 surviving queries
(the widths of a query group), row strides of 1, 2, 4 and more words, tables
wide enough for each group width, and long queries in a batch of short ones.
Every ID list equals the oracle's."""
import numpy as np
import pytest

import synth
from tests.parity import assert_query_equal

pytestmark = pytest.mark.gpu


def _collection(rng, lists):
    off = np.zeros(len(lists) + 1, np.uint64)
    np.cumsum([len(x) for x in lists], out=off[1:])
    return synth.Collection("keys", np.concatenate(lists), off)


@pytest.mark.parametrize("K,B,R,eta", [
    (1, 1, 1, 1), (31, 5, 2, 1), (255, 20, 3, 2), (256, 33, 8, 2), (257, 64, 6, 3), (2048, 100, 5, 4),
    (2049, 320, 8, 3), (4500, 1024, 8, 1), (6000, 4096, 8, 1), (140_001, 130, 4, 2)])
def test_probe_and_set_kernels_at_tile_edges(K, B, R, eta):
    import torch

    from oracle.oracle import Oracle
    from paper_1910_02611_gb300 import Plan, Rambo

    rng = np.random.default_rng(K + B)
    m = 1 << 12
    vocab = rng.integers(0, 1 << 63, 300, dtype=np.uint64)
    pop = 1.0 / np.arange(1, vocab.size + 1)
    pop /= pop.sum()
    ids = np.unique(np.concatenate([rng.choice(K, min(K, 1200), replace=False), [0, K - 1]])).astype(np.uint64)
    sets = _collection(rng, [np.unique(rng.choice(vocab, int(rng.integers(1, 30)), p=pop)) for _ in ids])
    g, o = Rambo(K, B, R, m, eta, 9), Oracle(K, B, R, m, eta, 9)
    g.insert(ids, sets.data, sets.offsets, kind="keys")
    o.insert_keys_batch(ids, sets.data, sets.offsets)

    def queries(n, most):
        return _collection(rng, [rng.choice(vocab, int(rng.integers(1, most + 1)), p=pop) for _ in range(n)])

    for n in (1, 31, 32, 33, 64, 65, 128, 129, 300):
        assert_query_equal(g, o, queries(n, 3))  # lane groups
    assert_query_equal(g, o, queries(7, 90))  # warp groups
    assert_query_equal(g, o, queries(20_000, 40).subset(np.arange(3000)))  # a warp each
    # mostly one term, three queries of many
    mixed = [rng.choice(vocab, 1, p=pop) for _ in range(400)]
    for t in (0, 123, 399):
        mixed[t] = rng.choice(vocab[:8], 33 + t, p=pop[:8] / pop[:8].sum())
    q = _collection(rng, mixed)
    ids_h, off_h = assert_query_equal(g, o, q)
    # the same batch from device memory, and through a plan sized for more
    ids_d, off_d = g.query(torch.from_numpy(q.data.view(np.int64)).cuda(),
                           torch.from_numpy(q.offsets.view(np.int64)).cuda(), kind="keys")
    assert np.array_equal(off_d.cpu().numpy().view(np.uint64), off_h)
    assert np.array_equal(ids_d.cpu().numpy().view(np.uint32), ids_h)
    plan = Plan(g, "keys", 1000, q.data.size, max(1, ids_h.size))
    for _ in range(2):
        plan.launch_host(q.data, q.offsets)
        ids_p, off_p = plan.wait()
        assert np.array_equal(off_p, off_h) and np.array_equal(ids_p, ids_h)
    plan.close()
    g.close()
