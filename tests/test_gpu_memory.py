"""Calls in little device memory: what a context only keeps for later calls
goes back to an allocation that finds no room.  Results are compared with the
oracle or with the same call in plenty of memory."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fb():
    from paper_0905_2203_gb300 import build as b
    b.build()
    from paper_0905_2203_gb300 import binding
    return binding


def random_cands(seed, k, n_types, size, bins):
    r = np.random.default_rng(seed)
    offs = np.arange(0, k * size + 1, size, dtype=np.int64)
    ct = r.integers(0, n_types, k * size).astype(np.uint16)
    b = np.asarray(bins, np.int32)[r.integers(0, len(bins), k * (size - 1))]
    return offs, ct, np.ascontiguousarray(b[:, 0]), np.ascontiguousarray(b[:, 1])


def test_recounts_of_an_append_find_the_entry_lists_room(fb):
    """Chunks half slow, half ten times faster: segments are cut by the mean
    rate, so many episodes run out of entry classes in the fast half and are
    counted again grid-wide, in a budget that holds that count's arrays but
    not the first count's entry lists beside them."""
    n, chunk, n_types = 120_000, 40_000, 6
    r = np.random.default_rng(3)
    gap = np.where(np.arange(n) % chunk < chunk // 2, 100, 10)
    tm = np.cumsum(r.integers(1, 2 * gap, n)).astype(np.int32)
    ty = r.integers(0, n_types, n).astype(np.uint16)
    cands = random_cands(6, 400, n_types, 4, [(0, 800), (400, 800)])
    ctx = fb.Context(0, hbm_budget_bytes=42 << 20)
    try:
        sess = ctx.session(fb.Cands(*cands), n_types)
        again = 0
        for i in range(0, n, chunk):
            sess.append(ty[i:i + chunk], tm[i:i + chunk])
            again += ctx.last_stats()["fallback_recounts"]
        got = sess.counts().astype(np.int64)
        sess.close()
    finally:
        ctx.close()
    want, _ = oracle.count_many(ty, tm, *cands)
    assert np.array_equal(got, want.astype(np.int64))
    assert again > 50
