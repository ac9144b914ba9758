"""Skip-N batches in device memory, whose size the device reads itself: a
handle's first large one after a small one (the packed buffer and the mask of
unresolved bases are then too small, grow, and the batch runs again), and
offsets that point outside the batch or come back, which are refused with the
lowest-numbered bad query.  Every ID list equals the oracle's."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

SKIP_N = 0x200


@pytest.fixture(scope="module")
def work(tmp_path_factory):
    from oracle.oracle import Oracle
    from paper_1910_02611_gb300 import Rambo

    w = synth.make("genome", 0.01, m=1 << 16)
    data = w.queries.data.copy()
    data[w.queries.offsets[:-1].astype(np.int64) + 5] = ord("N")  # one unresolved base a query
    path = str(tmp_path_factory.mktemp("skipn") / "index")
    g, o = Rambo(w.K, w.B, w.R, w.m, w.eta, w.seed), Oracle(w.K, w.B, w.R, w.m, w.eta, w.seed)
    g.insert(w.sets.ids, w.sets.data, w.sets.offsets, kind="seq")
    o.insert_seq_batch(w.sets.ids, w.sets.data, w.sets.offsets, 31)
    g.save(path)
    g.close()
    # a loaded handle has packed no sequence yet
    return lambda: Rambo.load(path), o, w.queries, synth.Collection("seq", data, w.queries.offsets)


def _device(g, data, off, k):
    import torch

    ids, offs = g.query(torch.from_numpy(data).cuda(), torch.from_numpy(off.view(np.int64)).cuda(), kind="seq", k=k)
    return ids.cpu().numpy().view(np.uint32), offs.cpu().numpy().view(np.uint64)


@pytest.mark.parametrize("k", [31, 31 | SKIP_N, 12 | SKIP_N])
def test_a_fresh_handle_grows(work, k):
    fresh, o, plain, q = work
    q = q if k & SKIP_N else plain
    g = fresh()
    some = 0
    for n in (1, 1000, 2, 999):
        part = q.subset(np.arange(n))
        want = o.query_batch("seq", part.data, part.offsets, k=k)
        ids, off = _device(g, part.data, part.offsets, k)
        assert np.array_equal(off, want[1]) and np.array_equal(ids, want[0])
        some += ids.size
    assert some or k != 31
    g.close()


def test_offsets_outside_the_batch_are_refused(work):
    from paper_1910_02611_gb300 import EBADSEQ, EINVAL, RamboError

    fresh, o, _, q = work
    g = fresh()
    k = 31 | SKIP_N
    one = q.subset(np.arange(1))
    _device(g, one.data, one.offsets, k)
    data, none = q.data[:2000].copy(), np.full(100, ord("N"), np.uint8)
    far = 4_000_000
    cases = [
        (np.array([40, far, 2]), data, EINVAL, 0),  # ends before it starts
        (np.array([0, 100, far, 300]), data, EINVAL, 2),  # a middle one past the end
        (np.array([0, 500, 100, 900]), data, EINVAL, 1),
        (np.array([400, 100, 300, 900]), data, EINVAL, 0),  # before the first
        (np.array([0, 200, 300, far, 900]), np.concatenate([data[:200], none, data[300:]]), EBADSEQ, 1),
        (np.array([0, 200, 230, far, 900]), data, EBADSEQ, 1),  # shorter than k
    ]
    for off, bases, code, item in cases:
        with pytest.raises(RamboError) as e:
            _device(g, bases, off.astype(np.uint64), k)
        assert e.value.code == code and e.value.item == item, (off, e.value)
    want = o.query_batch("seq", one.data, one.offsets, k=k)
    ids, off = _device(g, one.data, one.offsets, k)
    assert np.array_equal(off, want[1]) and np.array_equal(ids, want[0])
    g.close()


def test_the_mask_grows_by_itself(work):
    """After a large batch without a mask, a small and a large one with it."""
    fresh, o, plain, q = work
    g = fresh()
    for k, n in ((31, 1000), (31 | SKIP_N, 1), (31, 1000), (31 | SKIP_N, 1000), (31 | SKIP_N, 999), (31, 1000)):
        part = (q if k & SKIP_N else plain).subset(np.arange(n))
        want = o.query_batch("seq", part.data, part.offsets, k=k)
        ids, off = _device(g, part.data, part.offsets, k)
        assert np.array_equal(off, want[1]) and np.array_equal(ids, want[0])
    g.close()
