"""What the host code asks of the kernels, and where, on a runtime without a
GPU (two devices): a handle's kernels are set up on the handle's device
whichever is current."""
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
