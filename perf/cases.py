"""The calls that a user of the library makes, as cases that can be timed.

Streams are spike trains of the families that the tests and the benchmark use
(Poisson neurons, optional network bursts, embedded chains of neurons that
follow one another), drawn on the GPU from a seed.  Every pass goes through
the public binding.

Kinds of case:
  count    exact counts of a given candidate set over one resident stream
           (candidates and counts in host memory)
  mine     level-wise mining of resident recordings, all levels read back;
           `prepass` is the pre-pass setting of the context (0 = the default,
           2 = the level-2 pair bound only, so that every level-3 candidate is
           counted exactly)
  fresh    mining of a recording that has just arrived in pinned host memory:
           upload, mining, results, release
  session  a recording that grows by appends, exact counts after the last one
  serve    a queue of mining jobs through the serving loop
"""
import ctypes
import math

import numpy as np
import torch

from paper_0905_2203_gb300 import binding as fb

_BINS_MS = ((0, 5), (5, 10), (10, 15), (15, 20))
_ROOM = 30000  # 32-bit words of frequent episodes kept for a recording


def listed():
    return [
        # a short test recording and a few hundred candidates: all latency
        {"name": "count_tiny", "kind": "count", "n": 5003, "types": 32, "rate_lo": 5.0, "rate_hi": 5.0,
         "tick_us": 1000, "bursts": False, "cands": 512, "size_lo": 2, "size_hi": 4},
        # a handful of long episodes (hypotheses about one circuit) over a
        # long recording of a 64-neuron culture
        {"name": "count_few", "kind": "count", "n": 11000000, "types": 64, "rate_lo": 20.0, "rate_hi": 20.0,
         "tick_us": 100, "bursts": False, "cands": 16, "size_lo": 4, "size_hi": 8},
        # an ordinary candidate set over an ordinary recording
        {"name": "count_mid", "kind": "count", "n": 1071233, "types": 128, "rate_lo": 2.0, "rate_hi": 20.0,
         "tick_us": 1, "bursts": False, "cands": 3001, "size_lo": 2, "size_hi": 6},
        # batched counting: every candidate of a study over one bursty stream
        {"name": "count_large", "kind": "count", "n": 4000000, "types": 60, "rate_lo": 20.0, "rate_hi": 20.0,
         "tick_us": 10, "bursts": True, "cands": 200000, "size_lo": 2, "size_hi": 8},
        # mining a short test recording (half a minute of 32 neurons)
        {"name": "mine_tiny", "kind": "mine", "recs": 1, "n_lo": 5003, "n_hi": 5003, "types": 32, "rate_lo": 5.0,
         "rate_hi": 5.0, "tick_us": 1000, "thr": 0.01, "max_size": 4, "prepass": 0},
        # mining one ordinary recording (a quarter of an hour of 128 neurons)
        {"name": "mine_mid", "kind": "mine", "recs": 1, "n_lo": 1071233, "n_hi": 1071233, "types": 128,
         "rate_lo": 2.0, "rate_hi": 20.0, "tick_us": 1, "thr": 0.0025, "max_size": 6, "prepass": 0},
        # mining many recordings of all lengths in one call
        {"name": "mine_many", "kind": "mine", "recs": 64, "n_lo": 10000, "n_hi": 5000000, "types": 60,
         "rate_lo": 5.0, "rate_hi": 20.0, "tick_us": 10, "thr": 0.0025, "max_size": 6, "prepass": 0},
        # the same work with every level-3 candidate counted exactly
        {"name": "mine_many_exact", "kind": "mine", "recs": 48, "n_lo": 10000, "n_hi": 5000000, "types": 60,
         "rate_lo": 5.0, "rate_hi": 20.0, "tick_us": 10, "thr": 0.0025, "max_size": 6, "prepass": 2},
        # one ordinary recording from host memory to its frequent episodes
        {"name": "fresh_mid", "kind": "fresh", "n": 1000003, "types": 128, "rate_lo": 5.0, "rate_hi": 20.0,
         "tick_us": 10, "thr": 0.0025, "max_size": 6},
        # a long recording of a large array, from host memory
        {"name": "fresh_large", "kind": "fresh", "n": 20000000, "types": 256, "rate_lo": 20.0, "rate_hi": 30.0,
         "tick_us": 10, "thr": 0.003, "max_size": 6},
        # a recording followed while it is being made
        {"name": "session", "kind": "session", "n": 1000003, "types": 128, "rate_lo": 2.0, "rate_hi": 20.0,
         "tick_us": 1, "chunk": 100000, "cands": 256, "size_lo": 2, "size_hi": 5},
        # a queue of mining jobs of several sizes
        {"name": "serve", "kind": "serve", "jobs": 12, "n_lo": 50000, "n_hi": 2000000, "types_lo": 60,
         "types_hi": 256, "tick_us": 10, "thr_lo": 0.0025, "thr_hi": 0.01},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["count", "count", "few", "mine", "mine", "many", "fresh", "fresh", "session", "serve"])
    tick = rng.choice([1, 10, 100])
    if kind == "count":
        size_lo = rng.choice([1, 2, 3])
        return {"kind": "count", "n": _log(rng, 5000, 4000000), "types": _log(rng, 32, 128), "rate_lo": 5.0,
                "rate_hi": 20.0, "tick_us": tick, "bursts": rng.random() < 0.5, "cands": _log(rng, 257, 100000),
                "size_lo": size_lo, "size_hi": rng.randint(max(size_lo, 2), 8)}
    if kind == "few":
        size_lo = rng.randint(2, 6)
        return {"kind": "count", "n": _log(rng, 1100000, 11000000), "types": _log(rng, 32, 128), "rate_lo": 20.0,
                "rate_hi": 20.0, "tick_us": 100, "bursts": False, "cands": _log(rng, 1, 128), "size_lo": size_lo,
                "size_hi": rng.randint(size_lo, 8)}
    if kind in ("mine", "many"):
        n_lo = _log(rng, 5000, 2000000) if kind == "mine" else _log(rng, 5000, 50000)
        return {"kind": "mine", "recs": 1 if kind == "mine" else _log(rng, 2, 48), "n_lo": n_lo,
                "n_hi": n_lo if kind == "mine" else _log(rng, 200000, 4000000), "types": _log(rng, 60, 128),
                "rate_lo": 5.0, "rate_hi": 20.0, "tick_us": tick if kind == "mine" else 10,
                "thr": round(rng.uniform(0.0025, 0.01), 4), "max_size": rng.randint(4, 8),
                "prepass": rng.choice([0, 0, 2])}
    if kind == "fresh":
        return {"kind": "fresh", "n": _log(rng, 100000, 15000000), "types": _log(rng, 60, 256), "rate_lo": 10.0,
                "rate_hi": 25.0, "tick_us": 10, "thr": round(rng.uniform(0.003, 0.01), 4),
                "max_size": rng.randint(4, 8)}
    if kind == "session":
        n = _log(rng, 100000, 2000000)
        return {"kind": "session", "n": n, "types": _log(rng, 60, 128), "rate_lo": 2.0, "rate_hi": 20.0,
                "tick_us": tick, "chunk": max(2000, n // rng.randint(3, 30)), "cands": _log(rng, 16, 2048),
                "size_lo": rng.choice([1, 2]), "size_hi": rng.randint(2, 6)}
    return {"kind": "serve", "jobs": rng.randint(3, 20), "n_lo": _log(rng, 20000, 80000),
            "n_hi": _log(rng, 300000, 2000000), "types_lo": 60, "types_hi": rng.randint(64, 256), "tick_us": 10,
            "thr_lo": 0.003, "thr_hi": round(rng.uniform(0.005, 0.01), 4)}


# --------------------------------------------------------------------------
# inputs

def _burst_times(g, u, dur):
    """Maps u in [0, 1) to times in [0, dur) of an intensity that is 10 times
    higher inside bursts of 100 to 300 ms every 2 to 10 s."""
    k = int(dur / 2.1) + 4
    gap = 2.0 + 8.0 * torch.rand(k, generator=g, device="cuda", dtype=torch.float64)
    ln = 0.1 + 0.2 * torch.rand(k, generator=g, device="cuda", dtype=torch.float64)
    edge = torch.zeros(2 * k + 1, device="cuda", dtype=torch.float64)
    edge[1:] = torch.cumsum(torch.stack([gap, ln], 1).reshape(-1), 0)
    edge = torch.clamp(edge, max=dur)
    width = edge[1:] - edge[:-1]
    width[1::2] *= 10.0
    cum = torch.zeros(2 * k + 1, device="cuda", dtype=torch.float64)
    cum[1:] = torch.cumsum(width, 0)
    x = u * cum[-1]
    i = torch.clamp(torch.searchsorted(cum, x, right=True) - 1, max=2 * k - 1)
    gain = torch.where(i % 2 == 1, 10.0, 1.0)
    return edge[i] + (x - cum[i]) / gain


def _stream(g, n, types, rate_lo, rate_hi, tick_us, bursts=False, chains=3):
    """Types (int16, the bits of uint16) and times (int32 ticks) of n events on
    the GPU, and the chains of neurons planted in them."""
    rates = rate_lo + (rate_hi - rate_lo) * torch.rand(types, generator=g, device="cuda", dtype=torch.float64)
    per_s = float(rates.sum()) * (1.0 + 9.0 * 0.2 / 6.2 if bursts else 1.0)
    dur = n / per_s
    m = int(n * 1.01) + 64
    cum = torch.cumsum(rates, 0) / rates.sum()
    ty = torch.searchsorted(cum, torch.rand(m, generator=g, device="cuda", dtype=torch.float64), right=True)
    ty = torch.clamp(ty, max=types - 1)
    u = torch.rand(m, generator=g, device="cuda", dtype=torch.float64)
    tm = _burst_times(g, u, dur) if bursts else u * dur
    perm = torch.randperm(types, generator=g, device="cuda").tolist()
    all_ty, all_tm, planted, at = [ty], [tm], [], 0
    for c in range(chains):
        length = 4 + (c % 3)
        neurons = perm[at:at + length]
        at += length
        if len(neurons) < length:
            break
        planted.append(neurons)
        cur = tm[ty == neurons[0]]
        for e in range(length - 1):
            cur = cur[torch.rand(cur.numel(), generator=g, device="cuda") < 0.9]
            centre = 2.5e-3 + 5e-3 * ((c + e) % 4)
            cur = cur + centre - 1e-3 + 2e-3 * torch.rand(cur.numel(), generator=g, device="cuda",
                                                          dtype=torch.float64)
            all_ty.append(torch.full_like(cur, neurons[e + 1], dtype=torch.int64))
            all_tm.append(cur)
    key = torch.floor(torch.cat(all_tm) * (1e6 / tick_us)).to(torch.int64) * 65536 + torch.cat(all_ty)
    key = torch.unique(key)[:n]
    return (key % 65536).to(torch.int16).contiguous(), (key // 65536).to(torch.int32).contiguous(), planted


def _bins(tick_us):
    return [(a * 1000 // tick_us, b * 1000 // tick_us) for a, b in _BINS_MS]


def _cands(seed, count, types, size_lo, size_hi, bins, planted):
    """A candidate set in CSR form: distinct random types, a random bin per
    edge; one in twenty follows a planted chain as far as it reaches."""
    r = np.random.default_rng(seed)
    sizes = r.integers(size_lo, size_hi + 1, count)
    offs = np.zeros(count + 1, np.int64)
    offs[1:] = np.cumsum(sizes)
    wide = max(int(sizes.max()), 1)
    seq = np.empty((count, wide), np.int64)
    for k in range(wide):  # distinct types: draw again where a type repeats
        v = r.integers(0, types, count)
        while k:
            again = (seq[:, :k] == v[:, None]).any(1)
            if not again.any():
                break
            v[again] = r.integers(0, types, int(again.sum()))
        seq[:, k] = v
    for c in np.nonzero(r.random(count) < 0.05)[0]:
        ch = planted[c % len(planted)] if planted else []
        head = ch[: int(sizes[c])]
        rest = [int(x) for x in seq[c] if int(x) not in head]
        row = (head + rest)[: int(sizes[c])]
        seq[c, : len(row)] = row
    ty = seq[np.arange(wide)[None, :] < sizes[:, None]].astype(np.uint16)
    pick = r.integers(0, len(bins), int(offs[-1]) - count)
    b = np.asarray(bins, np.int32)
    return offs, ty, np.ascontiguousarray(b[pick, 0]), np.ascontiguousarray(b[pick, 1])


_contexts = {}
_servers = []


def _ctx(prepass=0):
    """One context per setting, kept for the life of the process."""
    if prepass not in _contexts:
        ctx = fb.Context(0)
        if prepass:
            ctx.set_tuning(prepass=prepass)
        _contexts[prepass] = ctx
    return _contexts[prepass]


def _server():
    if not _servers:
        _servers.append(fb.Server(0, hbm_budget_bytes=64 << 30, max_jobs=16))
    return _servers[0]


class _State:
    """A case's inputs; its resident streams are freed with it."""

    def __init__(self, **kw):
        self.streams = []
        self.__dict__.update(kw)

    def __del__(self):
        for s in self.streams:
            s.free()


def _sizes(case, seed, count):
    """Event counts spread evenly over the logarithm of the case's range."""
    lo, hi = math.log(case["n_lo"]), math.log(case["n_hi"])
    r = np.random.default_rng(seed)
    return [int(round(math.exp(lo + (hi - lo) * (i + 0.5) / count))) + int(r.integers(0, 16)) for i in range(count)]


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    kind, bins = case["kind"], _bins(case["tick_us"])
    if kind == "serve":
        jobs = []
        sizes = _sizes(case, seed, case["jobs"])
        for i in range(case["jobs"]):
            f = (7 * i) % case["jobs"] / max(case["jobs"] - 1, 1)
            nt = int(case["types_lo"] + (case["types_hi"] - case["types_lo"]) * f)
            ty, tm, _ = _stream(g, sizes[i], nt, 20.0, 30.0, case["tick_us"])
            frac = case["thr_lo"] + (case["thr_hi"] - case["thr_lo"]) * ((5 * i) % case["jobs"]) / case["jobs"]
            jobs.append((ty.cpu().numpy().view(np.uint16), tm.cpu().numpy(), nt, int(frac * len(ty)), 4 + i % 5))
        return _State(kind=kind, jobs=jobs, bins=bins, server=_server())
    if kind == "mine":
        ctx = _ctx(case["prepass"])
        st = _State(kind=kind, ctx=ctx, bins=bins, max_size=case["max_size"])
        st.thresholds = []
        for n in _sizes(case, seed, case["recs"]):
            ty, tm, _ = _stream(g, n, case["types"], case["rate_lo"], case["rate_hi"], case["tick_us"])
            torch.cuda.current_stream().synchronize()
            st.streams.append(ctx.load_stream(ty, tm, case["types"]))
            st.thresholds.append(max(20, int(case["thr"] * len(ty))))
        return st
    ty, tm, planted = _stream(g, case["n"], case["types"], case["rate_lo"], case["rate_hi"], case["tick_us"],
                              case.get("bursts", False))
    torch.cuda.current_stream().synchronize()
    if kind == "fresh":
        return _State(kind=kind, ctx=_ctx(), types=ty.cpu().pin_memory(), times=tm.cpu().pin_memory(),
                      n_types=case["types"], bins=bins, threshold=int(case["thr"] * len(ty)),
                      max_size=case["max_size"])
    csr = _cands(seed, case["cands"], case["types"], case["size_lo"], case["size_hi"], bins, planted)
    cands = fb.Cands(*csr)
    if kind == "session":
        chunks = [(ty[i:i + case["chunk"]].contiguous(), tm[i:i + case["chunk"]].contiguous())
                  for i in range(0, len(ty), case["chunk"])]
        torch.cuda.current_stream().synchronize()
        return _State(kind=kind, ctx=_ctx(), chunks=chunks, cands=cands, csr=csr, n_types=case["types"])
    st = _State(kind=kind, ctx=_ctx(), cands=cands, csr=csr)
    st.streams.append(st.ctx.load_stream(ty, tm, case["types"]))
    return st


# --------------------------------------------------------------------------
# one pass

def _levels(res, n_recs, max_size, n, parts):
    """Appends every level of every recording to parts (node types, edge
    bounds and counts of a recording's level one after another, 32-bit words)
    and writes the number of its episodes to n[level - 1, recording]."""
    k = fb.I64()
    p = [fb.VP() for _ in range(5)]
    refs = [ctypes.byref(x) for x in p]
    for r in range(n_recs):
        for level in range(1, max_size + 1):
            fb.check(fb.fem_result_level(res.h, r, level, ctypes.byref(k), *refs), "fem_result_level")
            m = k.value
            if m == 0:
                break
            n[level - 1, r] = m
            parts.append(np.frombuffer(ctypes.string_at(p[1], 2 * m * level), np.uint16).astype(np.int32))
            if level > 1:
                parts.append(np.frombuffer(ctypes.string_at(p[2], 4 * m * (level - 1)), np.int32))
                parts.append(np.frombuffer(ctypes.string_at(p[3], 4 * m * (level - 1)), np.int32))
            parts.append(np.frombuffer(ctypes.string_at(p[4], 4 * m), np.int32))


def _found(n, parts):
    """The episodes of all levels in one array, zeros after them (its length
    depends on the case alone unless far more is frequent than is usual)."""
    total = sum(len(a) for a in parts)
    flat = np.zeros(max(_ROOM * n.shape[1], total), np.int32)
    np.concatenate(parts, out=flat[:total])
    return {"n": n, "episodes": flat}


def run(st):
    if st.kind == "count":
        return st.ctx.count_episodes(st.streams[0], st.cands)
    if st.kind == "mine":
        res = st.ctx.mine_levelwise(st.streams, st.bins, st.thresholds, st.max_size)
        n, parts = np.zeros((st.max_size, len(st.streams)), np.int64), []
        _levels(res, len(st.streams), st.max_size, n, parts)
        res.free()
        return _found(n, parts)
    if st.kind == "fresh":
        s = st.ctx.load_stream(st.types, st.times, st.n_types)
        res = st.ctx.mine_levelwise([s], st.bins, [st.threshold], st.max_size)
        n, parts = np.zeros((st.max_size, 1), np.int64), []
        _levels(res, 1, st.max_size, n, parts)
        res.free()
        s.free()
        return _found(n, parts)
    if st.kind == "session":
        sess = st.ctx.session(st.cands, st.n_types)
        for ty, tm in st.chunks:
            sess.append(ty, tm)
        out = sess.counts()
        sess.close()
        return out
    ids = [st.server.submit(ty, tm, nt, st.bins, thr, ms) for ty, tm, nt, thr, ms in st.jobs]
    n, parts = np.zeros((8, len(ids)), np.int64), []
    for j, i in enumerate(ids):
        res, _ = st.server.wait(i)
        _levels(res, 1, st.jobs[j][4], n[:, j:j + 1], parts)
        res.free()
    return _found(n, parts)


def work(case):
    """Bytes: the streams, candidates and counts once (6 bytes an event, 2 a
    node, 8 an edge, 4 a count).  Operations: one per pair of a candidate and
    an event of one of its types, where the candidates are given; for mining,
    one per event and bin of the level-2 step at least."""
    kind = case["kind"]
    if kind in ("count", "session"):
        nodes = case["cands"] * (case["size_lo"] + case["size_hi"]) / 2
        return {"bytes": 6.0 * case["n"] + 10.0 * nodes + 12.0 * case["cands"],
                "flops": nodes * case["n"] / case["types"]}
    if kind == "fresh":
        return {"bytes": 6.0 * case["n"], "flops": 4.0 * case["n"]}
    count = case["recs"] if kind == "mine" else case["jobs"]
    n = float(sum(_sizes(case, 0, count)))
    return {"bytes": 6.0 * n, "flops": 4.0 * n}
