"""Device batches whose answers fill the handle's ID buffer to the last entry:
the answers that the gather laid out there are the ones returned.  The buffer
holds 64 IDs at first, and n + 1 plus an eighth once n did not fit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first", [1, 100, 9_000, 800_000, 8_000_000])
def test_answers_as_many_as_the_buffer_holds(first):
    import torch

    from paper_1910_02611_gb300 import Rambo

    g = Rambo(8, 4, 2, 1 << 10, 2, 3)
    key = np.array([12345], np.uint64)
    g.insert(np.array([5], np.uint64), key, np.array([0, 1], np.uint64), kind="keys")  # the one set there is

    def ask(n):  # n queries of one answer each
        ids, off = g.query(torch.full((n,), 12345, device="cuda"), torch.arange(n + 1, device="cuda"), kind="keys")
        assert torch.equal(off, torch.arange(n + 1, device="cuda"))
        assert ids.numel() == n and bool((ids == 5).all())

    room = 64 if first <= 64 else first + 1 + (first + 1) // 8
    for n in (first, room, room - 1, room + 1):
        ask(n)
    g.close()
