"""Device memory that queries and plans keep, on a runtime without a GPU: the
bitmaps and masks of a batch are bounded by a quarter of the free memory, the
masks of wide layouts (hundreds of times their bitmaps) among them, and a plan
that can be made without them is made."""
import numpy as np
import pytest

from tests.fakecuda import Fake

MIB = 1 << 20
ENOMEM = -4


@pytest.fixture(scope="module")
def fake():
    return Fake()


def _keys(n):
    return np.arange(n, dtype=np.uint64), np.arange(n + 1, dtype=np.uint64)


# 384 bytes of bitmap and 100 KB of masks a query; 250 KB of bitmap and 2 KB of masks
@pytest.mark.parametrize("K,B,R", [(3000, 50_000, 16), (2_000_000, 500, 8)])
@pytest.mark.parametrize("on_device", [False, True])
def test_a_batch_keeps_a_quarter_of_the_free_memory_at_most(fake, K, B, R, on_device):
    fake.budget(0, 64 << 30)
    h = fake.create(K, B, R, 64)
    base = fake.used()
    fake.budget(0, base + 8192 * MIB)
    for n in (100, 30_000, 70_000, 70_000):  # (the last two are cut into chunks when they come from the host)
        assert fake.query(h, *_keys(n), on_device) == 0
        assert fake.used() - base < 2048 * MIB + 64 * MIB, (n, fake.used() - base)
    fake.lib.rambo_destroy(h)


@pytest.mark.parametrize("K,B,R", [(3000, 50_000, 16), (2_000_000, 500, 8), (1000, 64, 4)])
def test_a_plan_keeps_a_quarter_of_the_free_memory_at_most_beside_what_it_needs(fake, K, B, R):
    """A plan of the query kernel alone shows what one needs in any case."""
    fake.budget(0, 64 << 30)
    h = fake.create(K, B, R, 64)
    cfg = _config(fake, h)
    for n, ids in ((1000, 1 << 20), (20_000, 1 << 27), (200_000, 1 << 27)):
        fake.budget(0, 64 << 30)
        cfg.set_stage, cfg.row_load = int(B > 4096), 0
        assert fake.lib.rambo_set_query_config(h, cfg) == 0
        base = fake.used()
        rc, p = fake.plan(h, 0, n, 4 * n, ids)
        assert rc == 0
        need = fake.used() - base
        fake.lib.rambo_plan_destroy(p)
        assert fake.used() == base
        cfg.set_stage, cfg.row_load = 0, 7
        assert fake.lib.rambo_set_query_config(h, cfg) == 0
        for room in (need, need + 100 * MIB, 3 * need, 64 << 30):
            fake.budget(0, base + room)
            rc, p = fake.plan(h, 0, n, 4 * n, ids)
            assert rc == 0, (n, ids, room, need)
            assert fake.used() - base <= need + room // 4, (n, ids, room, need, fake.used() - base)
            fake.lib.rambo_plan_destroy(p)
            assert fake.used() == base
        fake.budget(0, base + need - MIB)
        assert fake.plan(h, 0, n, 4 * n, ids)[0] == ENOMEM
        assert fake.used() == base
    fake.lib.rambo_destroy(h)


def test_a_skip_n_batch_does_not_allocate_a_mask_for_the_largest_batch_before_it(fake):
    fake.budget(0, 64 << 30)
    h = fake.create(1000, 64, 4, 64)
    data, ends = np.full(200_000_000, ord("A"), np.uint8), lambda n: np.array([0, n], np.uint64)
    for _ in range(2):
        assert fake.query(h, data, ends(data.size), True) == 0
    base = fake.used()
    for n in (400, 4000, 40_000):
        assert fake.query(h, data, ends(n), True, 31 | 0x200) == 0
    assert fake.used() - base < MIB
    fake.lib.rambo_destroy(h)


@pytest.mark.parametrize("R,m", [(1, 1 << 15), (5, 1 << 23)])  # 135 MB; 172 GB, more than 4096 windows of 8192 rows
def test_large_builds_are_bucketed_up_to_4096_windows_of_48_mib(fake, R, m):
    fake.budget(0, 280 << 30)
    h = fake.create(1000, 32_880, R, m, 2)  # rows of 4112 bytes: 12240 of them in a window
    n = -(-(1 << 26) // (2 * R)) + 1
    ids, keys, ends = np.zeros(1, np.uint64), np.zeros(n, np.uint64), np.array([0, n], np.uint64)
    fake.clear()
    fake.status(0, 2**64 - 1)
    assert fake.lib.rambo_insert_batch(h, ids.ctypes.data, keys.ctypes.data, ends.ctypes.data, 1, 0, None) == 0
    fake.status()
    names = [e["name"] for e in fake.events("L")]
    assert any("k_bucket_scatter" in x for x in names) and not any("k_insert" in x for x in names)
    assert sum("k_bucket_apply" in x for x in names) <= 4096
    fake.lib.rambo_destroy(h)


def _config(fake, h):
    from paper_1910_02611_gb300.rambo import QueryConfig

    cfg = QueryConfig()
    assert fake.lib.rambo_get_query_config(h, cfg) == 0
    return cfg
