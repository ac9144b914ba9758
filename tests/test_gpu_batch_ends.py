"""Batches whose start and end the device reads itself, and small host batches
that travel in one copy: a device batch larger than any before it (the packed
buffer grows and the batch runs again), offsets that start past zero, offsets
that end before they start, and host batches around the 64 KiB a copy takes.
Every ID list equals the oracle's."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pair():
    from oracle.oracle import Oracle
    from paper_1910_02611_gb300 import Rambo

    w = synth.make("genome", 0.01, m=1 << 16)
    g, o = Rambo(w.K, w.B, w.R, w.m, w.eta, w.seed), Oracle(w.K, w.B, w.R, w.m, w.eta, w.seed)
    g.insert(w.sets.ids, w.sets.data, w.sets.offsets, kind="seq")
    o.insert_seq_batch(w.sets.ids, w.sets.data, w.sets.offsets, 31)
    yield w, g, o
    g.close()


def _device(g, data, off, **kw):
    import torch

    d = torch.from_numpy(data if data.dtype == np.uint8 else data.view(np.int64)).cuda()
    ids, offs = g.query(d, torch.from_numpy(off.view(np.int64)).cuda(), **kw)
    return ids.cpu().numpy().view(np.uint32), offs.cpu().numpy().view(np.uint64)


@pytest.mark.parametrize("k", [31, 31 | 0x200])
def test_device_batches_that_grow_and_start_anywhere(pair, k):
    w, g, o = pair
    for n in (1, 3, 400, 40, 1000):  # 1, then far more than the packed buffer of the batch before
        q = w.queries.subset(np.arange(n))
        want = o.query_batch("seq", q.data, q.offsets, k=k)
        for lead in (0, 5, 64):
            data = np.concatenate([np.full(lead, ord("A"), np.uint8), q.data])
            ids, off = _device(g, data, q.offsets + np.uint64(lead), kind="seq", k=k)
            assert np.array_equal(off, want[1]) and np.array_equal(ids, want[0])
    keys = np.arange(300, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
    off = np.array([7, 9, 10, 60, 300], np.uint64)
    want = o.query_batch("keys", keys[7:], off - np.uint64(7))
    ids, offs = _device(g, keys, off, kind="keys")
    assert np.array_equal(offs, want[1]) and np.array_equal(ids, want[0])


def test_offsets_that_end_before_they_start(pair):
    from paper_1910_02611_gb300 import EINVAL, RamboError

    w, g, o = pair
    for kind, data in (("keys", np.arange(50, dtype=np.uint64)), ("seq", w.queries.data[:400])):
        with pytest.raises(RamboError) as e:
            _device(g, data, np.array([40, 45, 2], np.uint64), kind=kind)
        assert e.value.code == EINVAL and e.value.item == 0
    q = w.queries.subset(np.arange(20))
    want = o.query_batch("seq", q.data, q.offsets, k=31)
    ids, off = _device(g, q.data, q.offsets, kind="seq")
    assert np.array_equal(off, want[1]) and np.array_equal(ids, want[0])


@pytest.mark.parametrize("n", [1, 4094, 4095, 4096, 8190, 9000])
def test_host_batches_around_one_copy(pair, n):
    w, g, o = pair
    rng = np.random.default_rng(n)
    for per in (1, 7):
        keys = rng.integers(0, 1 << 62, n * per, dtype=np.uint64)
        off = np.arange(0, n * per + 1, per, dtype=np.uint64)
        ids, offs = g.query(keys, off, kind="keys")
        rids, roff = o.query_batch("keys", keys, off)
        assert np.array_equal(offs, roff) and np.array_equal(ids, rids)
