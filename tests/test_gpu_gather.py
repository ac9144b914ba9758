"""The gather's cut of long answers into parts: answers around 4096 IDs (not
cut up to there), bitmaps below and above 2048 words (a part's in a batch that
fills the grid), batches of a few queries (parts as short as 128 words) and of
many, ID lists and bitmaps, and answers that start at every offset of 16
bytes.  Every ID list equals the oracle's."""
import numpy as np
import pytest

import synth
from tests.parity import assert_query_equal

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,share", [(4097, 1.0), (40_000, 1.0), (70_001, 0.3), (140_001, 0.9)])
def test_long_answers_in_parts(K, share):
    from oracle.oracle import Oracle
    from paper_1910_02611_gb300 import Rambo

    rng = np.random.default_rng(K)
    g, o = Rambo(K, 40, 3, 1 << 8, 2, 4), Oracle(K, 40, 3, 1 << 8, 2, 4)
    few, many = rng.integers(0, 1 << 63, 6, dtype=np.uint64), rng.integers(0, 1 << 63, 2, dtype=np.uint64)
    ids = np.sort(rng.choice(K, max(4097, int(K * share)), replace=False)).astype(np.uint64)
    # every set holds the first of `many`, the first half of them the second, single sets one of `few` each
    lists = [many[: 1 + (2 * i < ids.size)] for i in range(ids.size)]
    for i, key in enumerate(few):
        at = int(rng.integers(0, ids.size))
        lists[at] = np.append(lists[at], key)
    off = np.zeros(ids.size + 1, np.uint64)
    np.cumsum([x.size for x in lists], out=off[1:])
    g.insert(ids, np.concatenate(lists), off, kind="keys")
    o.insert_keys_batch(ids, np.concatenate(lists), off)
    pool = [many[:1], many[1:], many, *(few[i : i + 1] for i in range(few.size)), rng.integers(0, 1 << 63, 3, dtype=np.uint64)]
    base = g.get_config()
    for staging in (0, 1):
        g.set_config(**{**base, "answer_staging": staging})
        for n in (1, 2, 9, 120):
            qs = [pool[int(i)] for i in rng.integers(0, len(pool), n)]
            qs[0] = pool[0]
            qo = np.zeros(n + 1, np.uint64)
            np.cumsum([x.size for x in qs], out=qo[1:])
            got, goff = assert_query_equal(g, o, synth.Collection("keys", np.concatenate(qs), qo))
            assert goff[1] - goff[0] >= 4097
    g.close()
