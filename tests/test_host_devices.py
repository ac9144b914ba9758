"""What the host code asks of the kernels, and where, on a runtime without a
GPU (two devices): a handle's kernels are set up on the handle's device
whichever is current, and the query that promises to load no code asks nothing
of kernels that creating the handle did not load."""
import numpy as np
import pytest

from tests.fakecuda import Fake


@pytest.fixture(scope="module")
def fake():
    f = Fake()
    yield f
    f.device(0)


@pytest.mark.parametrize("K,B,R", [(5000, 1000, 8), (5000, 20_000, 4), (300, 40, 3)])
@pytest.mark.parametrize("first", ["plan", "noalloc", "query"])
def test_a_handle_is_set_up_on_its_own_device(fake, K, B, R, first):
    fake.device(0)
    h = fake.create(K, B, R, 64)
    fake.device(1)  # the program's other GPU is current
    fake.clear()
    plan = None
    bases, ends = np.full(6200, ord("A"), np.uint8), np.arange(0, 6201, 31, dtype=np.uint64)
    if first == "plan":
        rc, plan = fake.plan(h, 0, 400, 4000, 1 << 20)
        assert rc == 0
    elif first == "noalloc":
        assert fake.noalloc(h, bases, ends) == 0
    assert fake.query(h, np.arange(200, dtype=np.uint64), np.arange(201, dtype=np.uint64), False) == 0
    assert fake.query(h, bases, ends, True) == 0
    events = fake.events()
    assert any("k_set" in e["name"] for e in events if e["kind"] == "L")
    assert all(e["device"] == 0 for e in events), [e for e in events if e["device"]]
    if plan:
        fake.lib.rambo_plan_destroy(plan)
    fake.lib.rambo_destroy(h)


@pytest.mark.parametrize("K,B,R,eta", [(5000, 1000, 8, 2), (5000, 20_000, 4, 1), (300, 40, 3, 3), (200_000, 64, 5, 4)])
def test_a_no_alloc_query_uses_only_kernels_that_creation_loaded(fake, K, B, R, eta):
    """Under lazy loading the first use of a kernel loads it, be it a question about its occupancy."""
    fake.device(0)
    fake.clear()
    h = fake.create(K, B, R, 64, eta)
    loaded = {e["name"] for e in fake.events("LF")}
    bases, ends = np.full(6200, ord("A"), np.uint8), np.arange(0, 6201, 31, dtype=np.uint64)
    for change in (None, "config", "fold", None):
        if change == "config":
            cfg = fake.config(h)
            cfg.visit_order = 1
            cfg.blocks_per_sm = 1
            assert fake.lib.rambo_set_query_config(h, cfg) == 0
        elif change == "fold":
            fake.clear()
            assert fake.lib.rambo_fold(h, None) == 0
            loaded |= {e["name"] for e in fake.events("LF")}
        for n in (200, 1):
            fake.clear()
            assert fake.noalloc(h, bases, ends[: n + 1]) == 0
            events = fake.events()
            assert any(e["kind"] == "L" for e in events)
            assert {e["name"] for e in events if e["name"]} <= loaded
            assert not any(e["kind"] == "M" for e in events)
        # what the no-alloc call resolved is not all that an ordinary query needs
        if change is None:
            assert fake.query(h, np.arange(2000, dtype=np.uint64), np.arange(2001, dtype=np.uint64), False) == 0
            assert any("k_set" in e["name"] for e in fake.events("L"))
    fake.lib.rambo_destroy(h)


@pytest.mark.parametrize("n,bases", [(1, 3_000_000), (7, 3_000_000), (1, 20_000_000), (300, 3_000_000)])
def test_long_sequences_on_the_device_are_packed_by_enough_blocks(fake, n, bases):
    fake.device(0)
    h = fake.create(300, 40, 3, 64)
    data, ends = np.full(bases, ord("A"), np.uint8), np.linspace(0, bases, n + 1).astype(np.uint64)
    for _ in range(2):  # (a handle's first sequences are sized on the host, later ones on the device)
        fake.clear()
        assert fake.query(h, data, ends, True) == 0
        (intake,) = [e for e in fake.events("L") if "k_intake" in e["name"]]
        assert intake["grid"] >= min(8 * 152, bases // 32 // 256), intake
    fake.lib.rambo_destroy(h)


@pytest.mark.parametrize("K", [10_000_000, 500_000_000])
def test_the_gather_of_one_answer_is_cut_into_a_bounded_number_of_parts(fake, K):
    """Every part counts its bitmap from the start, so their number is the number of times it is read."""
    fake.device(0)
    h = fake.create(K, 2000, 2, 64)
    for n in (1, 3):
        fake.clear()
        assert fake.query(h, np.arange(n, dtype=np.uint64), np.arange(n + 1, dtype=np.uint64), False) == 0
        (gather,) = [e for e in fake.events("L") if "k_gather" in e["name"]]
        assert gather["grid"] * 8 <= 128 * n + 8, gather  # (eight warps a block, a part each)
    fake.lib.rambo_destroy(h)


@pytest.mark.parametrize("K,parts", [(2000, 1), (2049, 2), (4000, 2), (8000, 4)])
def test_answers_over_a_few_thousand_sets_take_several_warps(fake, K, parts):
    """With one warp for each, 16 answers of 2000 IDs out of 4000 took 62 us through a plan, 52 before, now 39."""
    fake.device(0)
    h = fake.create(K, 64, 3, 64)
    fake.clear()
    assert fake.query(h, np.arange(64, dtype=np.uint64), np.arange(65, dtype=np.uint64), False) == 0
    (gather,) = [e for e in fake.events("L") if "k_gather" in e["name"]]
    assert gather["grid"] == 64 * parts // 8, gather
    fake.lib.rambo_destroy(h)


@pytest.mark.parametrize("n,terms,modes", [(2047, 1, "0"), (2048, 1, "2"), (2048, 8, "02"), (20_000, 9, "0"), (2048, 9, "1"), (300, 400, "1")])
def test_the_probe_instance_of_a_host_batch(fake, n, terms, modes):
    """0 a warp a query, 1 several warps, 2 lane groups (and a warp for the long ones, if there can be one)."""
    fake.device(0)
    h = fake.create(5000, 500, 4, 64)
    fake.clear()
    assert fake.query(h, np.arange(n * terms, dtype=np.uint64), np.arange(0, n * terms + 1, terms, dtype=np.uint64), False) == 0
    got = {e["name"].split("k_probeI")[1].split("EEEv")[0][-1] for e in fake.events("L") if "k_probeI" in e["name"]}
    assert got == set(modes), got
    fake.lib.rambo_destroy(h)
