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


def poisson_types(seed, n, n_types, per):
    """n events of n_types types at 5 to 20 units of rate, `per` ticks apart on
    average, sorted, no repeated (type, time)."""
    r = np.random.default_rng(seed)
    p = np.random.default_rng(7).uniform(5, 20, n_types)
    ty = r.choice(n_types, n, p=p / p.sum())
    key = np.unique(np.sort(r.integers(0, n * per, n)) * 65536 + ty)
    return (key % 65536).astype(np.uint16), (key // 65536).astype(np.int32)


def test_a_served_job_has_the_list_positions_room_after_level_2(fb):
    """A lone job whose third level needs, beside the recording, its lists and
    their index, more than what the budget leaves while the list positions
    (4 bytes an event) are kept; they are read by level 2 alone."""
    ty, tm = poisson_types(1, 4_080_000, 60, 83)
    bins, thr = [(0, 500), (500, 1000), (1000, 1500), (1500, 2000)], 8000
    srv = fb.Server(0, hbm_budget_bytes=128 << 20, max_jobs=2)
    try:
        res, _ = srv.wait(srv.submit(ty, tm, 60, bins, thr, 3), 120_000)
        got = [np.asarray(a) for k in (1, 2, 3) for a in res.level_arrays(0, k)]
        res.free()
    finally:
        srv.close()
    ctx = fb.Context(0)
    st = ctx.load_stream(ty, tm, 60)
    res = ctx.mine_levelwise([st], bins, [thr], 3)
    want = [np.asarray(a) for k in (1, 2, 3) for a in res.level_arrays(0, k)]
    res.free()
    st.free()
    ctx.close()
    assert all(np.array_equal(a, b) for a, b in zip(got, want)) and len(want[9]) > 0


@pytest.mark.parametrize("host_path", [False, True])
def test_loads_find_the_list_positions_room(fb, host_path):
    """Recordings arrive after a recording of 2M events was mined: as many find
    room as when it was only counted (mining keeps 8 MB of list positions for
    the next call, fourteen of the arriving recordings), and mined again it
    gives the same result."""
    a, b = poisson_types(2, 2_000_000, 60, 83), poisson_types(3, 100_000, 60, 83)
    bins = [(0, 500), (500, 1000)]

    def mine(ctx, s):
        res = ctx.mine_levelwise([s], bins, [20_000], 3)
        out = [np.asarray(x) for k in (1, 2, 3) for x in res.level_arrays(0, k)]
        res.free()
        return out

    def room(ctx):
        got = []
        with pytest.raises(fb.FemError) as e:
            while len(got) < 1000:
                got.append(ctx.load_stream(*b, 60))
        assert e.value.status == fb.FEM_ERR_NOMEM
        for x in got:
            x.free()
        return len(got)

    ctx = fb.Context(0, hbm_budget_bytes=80 << 20)
    s = ctx.load_stream(*a, 60)
    ctx.count_episodes(s, fb.Cands(*random_cands(5, 300, 60, 3, bins)))
    counted = room(ctx)
    ctx.close()
    ctx = fb.Context(0, hbm_budget_bytes=80 << 20)
    if host_path:
        ctx.set_tuning(level_graph=-1)
    s = ctx.load_stream(*a, 60)
    first = mine(ctx, s)
    mined = room(ctx)
    again = mine(ctx, s)
    ctx.close()
    assert mined >= counted - 7
    assert all(np.array_equal(x, y) for x, y in zip(first, again))


def test_frequent_sets_larger_than_the_packed_results(fb):
    """Frequent pairs of 256 recordings that pass the 64 MB of mapped results
    are read from the device arrays: the host-driven path's sets, level by
    level."""
    n_types, bins = 60, [(0, 2000), (2000, 4000), (4000, 6000), (6000, 8000)]
    data = [poisson_types(100 + r, 1200, n_types, 10) for r in range(256)]
    ctx = fb.Context(0)
    st = [ctx.load_stream(t, x, n_types) for t, x in data]

    def mine():
        res = ctx.mine_levelwise(st, bins, [0] * len(st), 2)
        out = [res.level_arrays(r, k) for r in range(len(st)) for k in (1, 2)]
        tails = res.stats()["graph_tails"]
        res.free()
        return out, tails

    try:
        got, tails = mine()
        ctx.set_tuning(level_graph=-1)
        want, _ = mine()
    finally:
        ctx.close()
    assert tails == 1
    assert sum(len(x[4]) for x in want[1::2]) * 20 > 64 << 20
    for a, b in zip(got, want):
        assert all(np.array_equal(x, y) for x, y in zip(a, b))


def test_counts_wherever_the_recording_fits(fb):
    """Once a budget holds a recording of 1M events and its candidates, every
    larger one counts: room for the per-type lists or their time index but not
    for what counting over them takes is no reason to refuse."""
    ty, tm = poisson_types(4, 1_000_000, 60, 83)
    r = np.random.default_rng(5)
    offs = np.concatenate([[0], np.cumsum(r.integers(2, 6, 200))]).astype(np.int64)
    ct = r.integers(0, 60, int(offs[-1])).astype(np.uint16)
    lo = (r.integers(0, 4, len(ct) - 200) * 500).astype(np.int32)
    cands = offs, ct, lo, (lo + 500).astype(np.int32)
    want, _ = oracle.count_many(ty, tm, *cands)
    done = []
    for kb in range(7_500, 24_000, 500):
        ctx = fb.Context(0, hbm_budget_bytes=kb << 10)
        try:
            st = ctx.load_stream(ty, tm, 60)
            got = ctx.count_episodes(st, fb.Cands(*cands)).astype(np.int64)
            assert np.array_equal(got, want.astype(np.int64)), kb
            done.append(kb)
        except fb.FemError as e:
            assert e.status == fb.FEM_ERR_NOMEM
        finally:
            ctx.close()
    assert done == list(range(done[0], 24_000, 500)), done
    assert done[0] <= 12_000  # (6 MB; its lists and their index take 8 MB more)


def test_pair_bound_without_room_for_list_positions(fb):
    """13 MB hold a recording of 1M events (6 MB) and its lists (4 MB), not
    their positions (4 MB): the pair bound looks back over the stream instead
    and drops the same candidates."""
    ty, tm = poisson_types(6, 1_000_000, 60, 83)
    bins, thr = [(0, 500), (500, 1000), (1000, 1500)], 3_000

    def mine(budget):
        ctx = fb.Context(0, hbm_budget_bytes=budget)
        try:
            res = ctx.mine_levelwise([ctx.load_stream(ty, tm, 60)], bins, [thr], 2)
            out = [np.asarray(x) for k in (1, 2) for x in res.level_arrays(0, k)]
            stats = res.stats()
            res.free()
            return out, stats
        finally:
            ctx.close()

    (got, a), (want, b) = mine(13 << 20), mine(0)
    assert all(np.array_equal(x, y) for x, y in zip(got, want))
    assert a["candidates_pruned"] == b["candidates_pruned"] > 0
    assert a["graph_tails"] == 0 and b["graph_tails"] == 1
