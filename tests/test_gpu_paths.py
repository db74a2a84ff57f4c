"""GPU parity at the sizes where a dispatch changes its path: every count is
compared bit by bit with the CPU oracle."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fb():
    from paper_0905_2203_gb300 import build as b
    b.build()
    from paper_0905_2203_gb300 import binding
    return binding


@pytest.fixture(scope="module")
def ctx(fb):
    c = fb.Context(0)
    yield c
    c.close()


@pytest.fixture(scope="module")
def mid():
    return synth.c2_mid()


def oracle_counts(ty, tm, offs, ct, lo, hi):
    c, _ = oracle.count_many(ty, tm, offs, ct, lo, hi)
    return c.astype(np.int64)


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("wide", [1, 15, 100])
def test_few_episodes_over_a_long_recording(fb, ctx, mid, wide, device):
    """At most 256 episodes over more than 2^20 events: segments while spans
    are narrow (wide 1), segments with the overflowing episodes recounted
    grid-wide (15: about 12 events of a type in the longest span), grid-wide
    at once (100)."""
    import torch
    s, cfg = mid
    st = ctx.load_stream(s.types, s.times, s.n_types)
    bins = [(a * wide, b * wide) for a, b in cfg["bins"]]
    offs, ct, lo, hi = synth.random_candidates(0xFE0200 + wide, 40, s.n_types, 1, 6, bins, s.chains, 0.5)
    want = oracle_counts(s.types, s.times, offs, ct, lo, hi)
    args = (offs, ct, lo, hi)
    if device:
        args = tuple(torch.from_numpy(a.view(np.int16) if a.dtype == np.uint16 else a).cuda() for a in args)
        torch.cuda.synchronize()
    got = ctx.count_episodes(st, fb.Cands(*args)).astype(np.int64)
    assert np.array_equal(got, want), np.nonzero(got != want)[0][:5]
    assert want.max() > 0
    st.free()


def pair_bounds(ty, tm, n_types, bins):
    """ub[a, b, k]: b-events with an a-event inside bin k before them."""
    ub = np.zeros((n_types, n_types, len(bins)), np.int64)
    per = [tm[ty == a].astype(np.int64) for a in range(n_types)]
    for a in range(n_types):
        for b in range(n_types):
            for k, (lo, hi) in enumerate(bins):
                first = np.searchsorted(per[a], per[b] - hi, side="left")
                last = np.searchsorted(per[a], per[b] - lo, side="left")
                ub[a, b, k] = int((last > first).sum())
    return ub


PAIR_BINS = {
    "one": [(0, 7)],
    "gaps": [(3, 9), (20, 21)],
    "overlap": [(0, 12), (5, 30), (29, 31)],
    "eight": [(4 * k, 4 * k + 4) for k in range(8)],
    "wide": [(0, 70000), (70000, 2**31 - 1)],
}


@pytest.mark.parametrize("host_path", [False, True])
@pytest.mark.parametrize("bins", sorted(PAIR_BINS))
@pytest.mark.parametrize("n,n_types,t_max", [(40, 16, 30), (3000, 17, 9000), (2600, 40, 700), (5000, 16, 2**31 - 2)])
def test_pair_bound_drops_what_its_definition_drops(fb, ctx, n, n_types, t_max, bins, host_path):
    """Level 2: the candidates that the pair bound drops are those whose
    number of (second, first inside the bin) events is at or below the
    threshold, for windows of 0.1 to 100 events, ties, gaps between bins,
    overlapping bins and a window that reaches the last possible time."""
    ty, tm = synth.tiny_random_stream(31, n, n_types, t_max)
    bl = PAIR_BINS[bins]
    thr = max(1, n // (4 * n_types))
    ub = pair_bounds(ty, tm, n_types, bl)
    freq = np.bincount(ty, minlength=n_types)
    pairs = (freq[:, None] > thr) & (freq[None, :] > thr) & ~np.eye(n_types, dtype=bool)
    want = int((pairs[:, :, None] & (ub <= thr)).sum())
    kept = int((pairs[:, :, None] & (ub > thr)).sum())
    st = ctx.load_stream(ty, tm, n_types)
    ctx.set_tuning(level_graph=-1 if host_path else 0)
    try:
        res = ctx.mine_levelwise([st], bl, [thr], 2)
    finally:
        ctx.reset_tuning()
    if res.stats()["graph_tails"] == 1 and kept == 0:
        want = 0  # a graph's statistics end before a level that counts nothing
    assert res.stats()["candidates_pruned"] == want
    assert res.stats()["candidates_counted"] == kept
    res.free()
    st.free()


@pytest.mark.parametrize("recs", [1, 3])
@pytest.mark.parametrize("size_lo,size_hi", [(1, 5), (3, 3), (2, 16)])
def test_large_sets_share_their_first_two_nodes(fb, ctx, size_lo, size_hi, recs):
    """Sets large enough to be sorted by their first two nodes (2^14 episodes,
    1e9 relevant events), of mixed sizes, over one and several recordings:
    counts in input order.  Ten types and two bins make groups far longer than
    one item holds."""
    n_types, n_cand = 10, 21_000
    r = synth.Rng(5, size_hi)
    streams = [synth.tiny_random_stream(40 + i, 160_000 - 40_000 * i, n_types, 1_300_000) for i in range(recs)]
    sizes = r.integers(size_lo, size_hi, n_cand)
    offs = np.zeros(n_cand + 1, np.int64)
    offs[1:] = np.cumsum(sizes)
    ct = r.integers(0, n_types - 1, int(offs[-1])).astype(np.uint16)
    pick = r.integers(0, 1, int(offs[-1]) - n_cand)
    lo, hi = np.array([0, 9], np.int32)[pick], np.array([30, 55], np.int32)[pick]
    rec = r.integers(0, recs - 1, n_cand).astype(np.uint32)
    st = [ctx.load_stream(ty, tm, n_types) for ty, tm in streams]
    got = ctx.count_batch(st, fb.Cands(offs, ct, lo, hi), rec).astype(np.int64)
    for i, (ty, tm) in enumerate(streams):
        which = np.nonzero(rec == i)[0]
        so = np.zeros(len(which) + 1, np.int64)
        so[1:] = np.cumsum(sizes[which])
        nodes = np.concatenate([np.arange(offs[c], offs[c + 1]) for c in which])
        edges = np.concatenate([np.arange(offs[c] - c, offs[c + 1] - c - 1) for c in which])
        want = oracle_counts(ty, tm, so, ct[nodes], lo[edges], hi[edges])
        assert np.array_equal(got[which], want), np.nonzero(got[which] != want)[0][:5]
    assert got.max() > 0
    for s in st:
        s.free()


@pytest.mark.parametrize("t_max", [2_000, 40_000, 900_000])
@pytest.mark.parametrize("n", [31, 33, 64, 1000, 30_000])
def test_inner_nodes_by_entries(fb, ctx, n, t_max):
    """Inner nodes stepped by entries (forced), from 0.2 to 100 events of a
    type inside an edge, with chunks of entries that end a warp's 32."""
    n_types = 4
    ty, tm = synth.tiny_random_stream(60, n, n_types, t_max)
    r = synth.Rng(61, n)
    n_cand = 200
    sizes = r.integers(3, 6, n_cand)
    offs = np.zeros(n_cand + 1, np.int64)
    offs[1:] = np.cumsum(sizes)
    ct = r.integers(0, n_types - 1, int(offs[-1])).astype(np.uint16)
    lo = r.integers(0, 40, int(offs[-1]) - n_cand).astype(np.int32)
    hi = (lo + 1 + r.integers(0, 60, lo.size)).astype(np.int32)
    want = oracle_counts(ty, tm, offs, ct, lo, hi)
    st = ctx.load_stream(ty, tm, n_types)
    ctx.set_tuning(track_last=2)
    try:
        got = ctx.count_episodes(st, fb.Cands(offs, ct, lo, hi)).astype(np.int64)
    finally:
        ctx.reset_tuning()
    assert np.array_equal(got, want), np.nonzero(got != want)[0][:5]
    st.free()


def test_many_recordings_capture_again_when_a_level_overflows(fb, ctx):
    """Eight recordings in which every ordered pair survives level 2, four
    times what the first capture holds: the call captures a larger graph and
    finishes in it, with the host-driven path's results."""
    n_types, bins = 32, [(0, 50), (50, 100), (100, 150), (150, 200)]
    st = [ctx.load_stream(*synth.tiny_random_stream(0xCB0 + i, 40_000 + 1000 * i, n_types, 400_000), n_types)
          for i in range(8)]
    thr = [100] * 8

    def run():
        res = ctx.mine_levelwise(st, bins, thr, 2)
        out = [res.level(r, N) for r in range(8) for N in (1, 2)]
        stats = res.stats()
        res.free()
        return out, stats

    a, sa = run()
    ctx.set_tuning(level_graph=-1)
    try:
        h, _ = run()
    finally:
        ctx.reset_tuning()
    assert a == h
    assert sum(len(c) for _, c in h[1::2]) > 8 * n_types * (n_types - 1)
    assert sa["graph_tails"] == 1
    for s in st:
        s.free()


@pytest.mark.parametrize("chunk", [1, 700, 40_000])
@pytest.mark.parametrize("wide", [1, 12, 200])
def test_session_counts_by_segments_and_grid_wide(fb, ctx, wide, chunk):
    """Appends counted in segments (edges of up to 20 ticks; with 40,000-event
    chunks several segments), with episodes that run out of entry classes
    (240), and grid-wide or unsegmented (4000): after every append that is
    checked the counts are the oracle's on the prefix."""
    n_types = 6
    ty, tm = synth.tiny_random_stream(77, 90_000 if chunk > 1 else 2_000, n_types, 600_000 if chunk > 1 else 9_000)
    r = synth.Rng(78, wide)
    n_cand = 150
    sizes = r.integers(1, 5, n_cand)
    offs = np.zeros(n_cand + 1, np.int64)
    offs[1:] = np.cumsum(sizes)
    ct = r.integers(0, n_types - 1, int(offs[-1])).astype(np.uint16)
    lo = (r.integers(0, 9, int(offs[-1]) - n_cand) * wide).astype(np.int32)
    hi = (lo + wide * r.integers(1, 11, lo.size)).astype(np.int32)
    sess = ctx.session(fb.Cands(offs, ct, lo, hi), n_types)
    cuts = [0, 300, 301] + list(range(301 + chunk, min(len(ty), 301 + 40 * chunk), chunk)) + [len(ty)]
    try:
        for i, (a, b) in enumerate(zip(cuts[:-1], cuts[1:])):
            sess.append(ty[a:b], tm[a:b])
            if i < 4 or b == len(ty):
                want = oracle_counts(ty[:b], tm[:b], offs, ct, lo, hi)
                got = sess.counts().astype(np.int64)
                assert np.array_equal(got, want), (b, np.nonzero(got != want)[0][:5])
        assert want.max() > 0
        # relevant events of the last append: its recording's, tail included
        seen, _ = sess.info()
        assert seen == len(ty) and ctx.last_stats()["relevant_events"] > 0
    finally:
        sess.close()


@pytest.mark.parametrize("n_cand", [1, 33, 1025, 16_383, 16_384])
def test_one_recording_from_host_memory(fb, ctx, n_cand):
    """The short way of a host call (up to 16,383 episodes) and the general
    one: sizes 1-16, prefixes shared by runs longer than a group, one and many
    segments, counts to the host and to the device, the relaxed bound, and a
    malformed episode at the end refused with the counts untouched."""
    import torch
    n_types = 20
    r = synth.Rng(91, n_cand)
    sizes = np.repeat(r.integers(1, 16, (n_cand + 99) // 100), 100)[:n_cand]
    offs = np.zeros(n_cand + 1, np.int64)
    offs[1:] = np.cumsum(sizes)
    ct = r.integers(0, n_types - 1, int(offs[-1])).astype(np.uint16)
    lo = r.integers(0, 3, int(offs[-1]) - n_cand).astype(np.int32) * 10
    hi = lo + 25
    for c in range(1, n_cand):  # runs of 100 share all but their last node and edge
        if c % 100 and sizes[c] > 1:
            n = int(sizes[c])
            o, b = int(offs[c]), int(offs[c - 1])
            ct[o:o + n - 1] = ct[b:b + n - 1]
            lo[o - c:o - c + n - 2] = lo[b - c + 1:b - c + 1 + n - 2]
    hi = lo + 25
    for n_ev, t_max in ((3000, 9000), (60_000, 900_000)):
        ty, tm = synth.tiny_random_stream(92, n_ev, n_types, t_max)
        st = ctx.load_stream(ty, tm, n_types)
        want = oracle_counts(ty, tm, offs, ct, lo, hi)
        cands = fb.Cands(offs, ct, lo, hi)
        assert np.array_equal(ctx.count_episodes(st, cands).astype(np.int64), want)
        out = torch.zeros(n_cand, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        ctx.count_episodes(st, cands, out)
        assert np.array_equal(out.cpu().numpy().astype(np.int64), want)
        assert np.array_equal(ctx.upper_bound(st, cands).astype(np.int64),
                              oracle_counts(ty, tm, offs, ct, np.zeros_like(lo), hi))
        freq = np.bincount(ty, minlength=n_types)
        ctx.count_episodes(st, cands)
        assert ctx.last_stats()["relevant_events"] == freq[ct].sum()
        bad = ct.copy()
        bad[-1] = n_types
        keep = np.full(n_cand, 7, np.uint32)
        with pytest.raises(fb.FemError) as e:
            ctx.count_episodes(st, fb.Cands(offs, bad, lo, hi), keep)
        assert e.value.status == fb.FEM_ERR_INVAL and (keep == 7).all()
        st.free()


@pytest.mark.parametrize("recs,budget_mb", [(1, 28), (9, 40)])
def test_mining_in_little_memory(fb, ctx, mid, recs, budget_mb):
    """A budget that holds the recordings, their lists and one level, but not
    the list positions beside them."""
    s, cfg = mid
    n = s.n // recs
    cut = [(s.types[i * n:(i + 1) * n].copy(), s.times[i * n:(i + 1) * n].copy()) for i in range(recs)]
    thr = [cfg["threshold"] // recs] * recs

    def mine(c):
        st = [c.load_stream(t, x, s.n_types) for t, x in cut]
        res = c.mine_levelwise(st, cfg["bins"], thr, 5)
        out = [np.asarray(a) for r in range(recs) for k in range(1, 6) for a in res.level_arrays(r, k)]
        res.free()
        for x in st:
            x.free()
        return out

    small = fb.Context(0, hbm_budget_bytes=budget_mb << 20)
    try:
        got = mine(small)
    finally:
        small.close()
    want = mine(ctx)
    assert len(got) == len(want) and all(np.array_equal(a, b) for a, b in zip(got, want))


@pytest.mark.parametrize("n_cand,chunk,n_types,grid", [(8, 100_000, 2, True), (8, 5_000, 2, False),
                                                       (40, 60_000, 60, False)])
def test_wide_appends_take_the_shorter_way(fb, ctx, n_cand, chunk, n_types, grid):
    """Appends whose spans hold too many events of a type to cut the chunk: few
    episodes over long lists are counted grid-wide (no launch over work items),
    short lists by one warp an episode; counts are the oracle's either way."""
    ty, tm = synth.tiny_random_stream(79, 2 * chunk, n_types, 20 * chunk)
    wide = 10 * n_types * 12  # twelve events of a type per edge
    r = synth.Rng(80, n_cand)
    offs = np.arange(0, 4 * n_cand + 1, 4, dtype=np.int64)
    ct = r.integers(0, n_types - 1, 4 * n_cand).astype(np.uint16)
    lo = (r.integers(0, 1, 3 * n_cand) * wide // 2).astype(np.int32)
    hi = (lo + wide).astype(np.int32)
    sess = ctx.session(fb.Cands(offs, ct, lo, hi), n_types)
    try:
        for a in (0, chunk):
            sess.append(ty[a:a + chunk], tm[a:a + chunk])
            assert (ctx.last_stats()["sparse_launches"] == 0) == grid
        got = sess.counts().astype(np.int64)
    finally:
        sess.close()
    n = min(len(ty), 2 * chunk)
    want = oracle_counts(ty[:n], tm[:n], offs, ct, lo, hi)
    assert np.array_equal(got, want) and want.max() > 0


def test_captures_follow_what_calls_of_a_shape_needed(fb):
    """Eight short recordings: after a first call that needed little, the next
    is captured with the single-block kernels of small levels (fewer launches);
    one that needs far more is captured again; results are the host-driven
    path's throughout."""
    n_types, bins = 60, [(0, 50), (50, 100), (100, 150), (150, 200)]
    ctx = fb.Context(0)

    def mine(st, thr):
        res = ctx.mine_levelwise(st, bins, [thr] * 8, 3)
        out = [res.level(r, N) for r in range(8) for N in (1, 2, 3)]
        stats = res.stats()
        res.free()
        return out, stats

    try:
        launches = []
        for seed, thr in ((0, 60), (1, 60), (2, 4), (3, 60), (4, 4)):
            st = [ctx.load_stream(*synth.tiny_random_stream(0xCC0 + 16 * seed + i, 5000 + i, n_types, 100_000), n_types)
                  for i in range(8)]
            (a, s), (b, _) = mine(st, thr), mine(st, thr)
            launches.append(s["kernel_launches"])
            ctx.set_tuning(level_graph=-1)
            h, _ = mine(st, thr)
            ctx.reset_tuning()
            assert a == h and b == h and s["graph_tails"] == 1
            if thr == 4:
                assert sum(len(c) for _, c in h[1::3]) > 4096
            for x in st:
                x.free()
        assert launches[1] < launches[0]
    finally:
        ctx.close()


@pytest.mark.parametrize("force", [0, 2])
@pytest.mark.parametrize("rare,wide", [(1, 100_000), (3, 900), (40, 340), (40, 3_000), (700, 330)])
def test_entries_that_serve_many_events(fb, ctx, rare, wide, force):
    """A rare type followed by frequent ones at a wide edge: intervals of 15 to
    5,000 events, cut by the next entry or by the edge, at both ends of a
    chunk of entries; three to five nodes."""
    n, n_types = 30_000, 6
    ty, tm = synth.tiny_random_stream(95, n, n_types, 20 * n)
    r = synth.Rng(96, rare)
    ty = np.where(ty == 0, 1, ty)
    ty[r.integers(0, len(ty) // 3, rare)] = 0
    ok = np.concatenate([[True], np.diff(tm.astype(np.int64)) > 0])
    ty, tm = ty[ok].astype(np.uint16), tm[ok]
    n_cand = 120
    sizes = r.integers(3, 5, n_cand)
    offs = np.zeros(n_cand + 1, np.int64)
    offs[1:] = np.cumsum(sizes)
    ct = r.integers(1, n_types - 1, int(offs[-1])).astype(np.uint16)
    ct[offs[:-1]] = 0
    lo = r.integers(0, 30, int(offs[-1]) - n_cand).astype(np.int32)
    hi = (lo + 1 + r.integers(0, wide, lo.size)).astype(np.int32)
    hi[offs[:-1] - np.arange(n_cand)] += wide
    want = oracle_counts(ty, tm, offs, ct, lo, hi)
    st = ctx.load_stream(ty, tm, n_types)
    ctx.set_tuning(track_last=force)
    try:
        got = ctx.count_episodes(st, fb.Cands(offs, ct, lo, hi)).astype(np.int64)
    finally:
        ctx.reset_tuning()
    assert np.array_equal(got, want), np.nonzero(got != want)[0][:5]
    assert want.max() > 0
    st.free()


@pytest.mark.parametrize("host_path", [False, True])
@pytest.mark.parametrize("bins", ["eight", "overlap", "gaps"])
@pytest.mark.parametrize("n,n_types", [(33, 16), (700, 300), (5000, 900), (41_000, 500)])
def test_pair_bound_over_few_events_of_many_types(fb, ctx, n, n_types, bins, host_path):
    """Chunks of 32 list positions and four events a warp: lists of a few
    events, chunks that end inside one."""
    ty, tm = synth.tiny_random_stream(33, n, n_types, 3 * n)
    bl, thr = PAIR_BINS[bins], max(1, n // (2 * n_types))
    freq = np.bincount(ty, minlength=n_types)
    keep = np.nonzero(freq > thr)[0]
    ub = np.zeros((n_types, n_types, len(bl)), np.int64)
    for k, (lo, hi) in enumerate(bl):  # pairs of (b event, type) with an event of it in the window
        first = np.searchsorted(tm, tm.astype(np.int64) - hi, side="left")
        last = np.searchsorted(tm, tm.astype(np.int64) - lo, side="left")
        for j in range(len(tm)):
            ub[np.unique(ty[first[j]:last[j]]), ty[j], k] += 1
    pairs = np.zeros((n_types, n_types), bool)
    pairs[np.ix_(keep, keep)] = True
    np.fill_diagonal(pairs, False)
    kept = int((pairs[:, :, None] & (ub > thr)).sum())
    st = ctx.load_stream(ty, tm, n_types)
    ctx.set_tuning(level_graph=-1 if host_path else 0)
    try:
        res = ctx.mine_levelwise([st], bl, [thr], 2)
    finally:
        ctx.reset_tuning()
    assert res.stats()["candidates_counted"] == kept
    res.free()
    st.free()


JOIN_BINS = {
    "five": [(6 * k, 6 * k + 6) for k in range(5)],
    "eight": [(4 * k, 4 * k + 4) for k in range(8)],
    "gaps": [(3, 9), (14, 15), (20, 31)],
    "overlap": [(0, 12), (5, 30), (29, 31)],
    "overlap_six": [(0, 12), (2, 5), (5, 30), (8, 9), (29, 31), (30, 33)],
}


@pytest.mark.parametrize("bins", sorted(JOIN_BINS))
@pytest.mark.parametrize("recs", [1, 3])
def test_join_bound_over_any_bins(fb, ctx, recs, bins):
    """Level 3 with the join bound over five and more, gapped and overlapping
    bins: the oracle miner's sets, and fewer exact counts than without it."""
    n_types, bl = 16, JOIN_BINS[bins]
    thr = [{"five": 27, "eight": 19, "overlap": 60}.get(bins, 15)] * recs
    data = []
    for i in range(recs):
        ty, tm = synth.tiny_random_stream(0xB1 + i, 2600 + 64 * i, n_types, 5200)
        first = tm[ty == 0].astype(np.int64)  # a planted chain 0 -> 1 -> 2, seven ticks each
        key = np.unique(np.concatenate([tm.astype(np.int64) * 16 + ty, (first + 7) * 16 + 1, (first + 14) * 16 + 2]))
        data.append(((key % 16).astype(np.uint16), (key // 16).astype(np.int32)))
    st = [ctx.load_stream(ty, tm, n_types) for ty, tm in data]

    def mine():
        res = ctx.mine_levelwise(st, bl, thr, 3)
        out = [res.level(r, N) for r in range(recs) for N in (1, 2, 3)]
        stats = res.stats()
        res.free()
        return out, stats

    mine()  # (the first run may find a level larger than its capture)
    got, bounded = mine()
    ctx.set_tuning(prepass=2)
    try:
        mine()
        plain, exact = mine()
    finally:
        ctx.reset_tuning()
    for r, (ty, tm) in enumerate(data):
        want = oracle.mine_levelwise(ty, tm, n_types, bl, thr[r], 3)
        for N in (1, 2, 3):
            assert list(zip(*got[3 * r + N - 1])) == want[N], (r, N)
    assert plain == got
    assert bounded["graph_tails"] == exact["graph_tails"] == 1 and len(got[2][0]) > 0
    assert bounded["candidates_counted"] < exact["candidates_counted"]
    for s in st:
        s.free()


@pytest.mark.parametrize("hi,route", [(20, "segments"), (700, "recounts"), (9_000, "grid")])
def test_few_episodes_routes(fb, ctx, hi, route):
    """At most 256 episodes over more than 2^20 events, half of them ten times
    denser: segments; segments with episodes that run out of entry classes in
    the dense half and are counted again; grid-wide at once."""
    n, n_types = 1_100_000, 8
    r = np.random.default_rng(12)
    tm = np.cumsum(r.integers(1, np.where(np.arange(n) < n // 2, 200, 20))).astype(np.int32)
    ty = r.integers(0, n_types, n).astype(np.uint16)
    offs = np.arange(0, 4 * 30 + 1, 4, dtype=np.int64)
    ct = r.integers(0, n_types, 4 * 30).astype(np.uint16)
    lo = (r.integers(0, 2, 3 * 30) * hi // 2).astype(np.int32)
    up = np.full(3 * 30, hi, np.int32)
    st = ctx.load_stream(ty, tm, n_types)
    got = ctx.count_episodes(st, fb.Cands(offs, ct, lo, up)).astype(np.int64)
    s = ctx.last_stats()
    st.free()
    assert np.array_equal(got, oracle_counts(ty, tm, offs, ct, lo, up)) and got.max() > 0
    assert (s["sparse_launches"] == 0) == (route == "grid")
    assert (s["fallback_recounts"] > 0) == (route == "recounts")
