"""The bucketed construction's scatter and apply over their instances: one to
four hashes, up to eight tables and more, one, two and four keys a thread, one
window and several, row strides whose windows are not a power of two of rows,
keys that repeat (hot words) and keys that do not, and items from empty to
longer than a block's step.  The index equals, bit for bit, the one-pass
build's, and its per-cell population counts equal the oracle's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,R,m,eta,repeats", [
    (20, 2, 1 << 23, 1, False), (128, 8, 1 << 20, 4, True), (640, 5, 1 << 18, 3, True), (100, 9, 1 << 18, 3, False),
    (64, 16, 1 << 20, 2, True), (33, 12, 1 << 17, 1, False), (300, 7, 1 << 18, 2, True)])
def test_bucketed_build_instances(B, R, m, eta, repeats):
    from oracle.oracle import Oracle
    from paper_1910_02611_gb300 import Rambo

    rng = np.random.default_rng(B * R)
    K = 700
    sizes = rng.choice([0, 1, 2, 3, 40, 700, 5000], K, p=[0.2, 0.2, 0.1, 0.1, 0.2, 0.17, 0.03])
    sizes[:3], sizes[-3:] = 0, 0
    ids = rng.permutation(K).astype(np.uint64)
    off = np.zeros(K + 1, np.uint64)
    np.cumsum(sizes, out=off[1:])
    n = int(off[-1])
    keys = rng.integers(0, 1 << 63, n, dtype=np.uint64)
    if repeats:  # two keys in five are one of three
        hot = rng.random(n) < 0.4
        keys[hot] = keys[rng.integers(0, 3, int(hot.sum()))]
    built = []
    for mode in (3, 2):
        g = Rambo(K, B, R, m, eta, 11)
        g.set_build_tiling(mode=mode)
        g.insert(ids, keys, off, kind="keys")
        built.append((g.export_index(), g.cell_popcount(), g.export_registered()))
        g.close()
    for a, b in zip(*built):
        assert np.array_equal(a, b)
    o = Oracle(K, B, R, m, eta, 11)
    o.insert_keys_batch(ids, keys, off, nthreads=8)
    assert np.array_equal(built[0][1], o.cell_popcount())
