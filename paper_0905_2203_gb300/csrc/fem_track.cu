// fem_track.cu -- exact counting by node-by-node local tracking, one warp per
// (episode, segment) work item, in one persistent launch fed by an atomic
// work queue.
//
// The count is the size of the largest set of non-overlapped occurrences,
// found by Algorithm 1 ("Problem decomposition") over end events, each with
// the LATEST start of an occurrence ending there:
//     L_1(j) = t_j,   L_k(j) = max { L_{k-1}(i) : lo < t_j - t_i <= hi }.
// Over the events of node k-1 that have a valid L (the node's entries), L is
// non-decreasing in time, so L_k(j) is the L of the newest entry older than
// t_j - lo, provided that entry is not older than t_j - hi.  Section
// "Parallel Local Tracking" tracks an episode node by node over the per-type
// event lists; here one warp does that for one work item:
//   * node k's events (its type's list, inside the segment and its halo) are
//     taken 32 at a time, one per lane, in time order;
//   * each lane finds its predecessor among node k-1's entries with a window
//     walk: the warp loads 32 consecutive entries, every lane ranks its own
//     query in them by a 5-step binary search over the lanes' registers, and
//     the window moves on until every lane has its rank; queries of a node
//     come in time order, so the window only moves forward;
//   * the lanes that found a valid predecessor append (t, L) to the node's
//     entry list in the warp's buffer (ballot + prefix count);
//   * where the previous node's entries are the shorter side, the lanes take
//     32 of them instead and look up the events that each one serves with the
//     stream's per-type time index (inner_by_entries, last_by_entries);
//   * at the last node the valid ends inside the segment are handed, in time
//     order, to Algorithm 1 for every entry class of the segment (one class
//     per lane; the record is that of the other counting kernels, so k_stitch
//     composes the segments; section "MapConcat").
// Every lane of the warp does the same work on the same list, so lanes stay
// converged, list reads are coalesced and no per-node ring is needed: the
// entry lists live in a per-warp global buffer of 4 x (longest list) words.
//
// The launch is persistent: each warp takes the next item index from a
// counter until the items run out, so items of very different lengths (long
// and short recordings, short and long episodes) balance across the GPU.
#include <algorithm>

#include "fem_internal.cuh"

namespace fem {

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

// First i in [lo, hi) with v[i] >= q (hi if none), computed by the whole warp
// (every lane returns it): a 32-way search whose probes are one strided load.
// (Positions fit 32 bits: a recording has fewer than 2^30 events.)
__device__ __forceinline__ int warp_lower_bound(const int32_t *__restrict__ v, int lo, int hi, int32_t q, int lane) {
    while (hi - lo > 32) {
        const int step = (hi - lo + 31) >> 5;
        const int pos = lo + step * (lane + 1) - 1;
        const bool below = pos < hi && v[pos] < q;
        const int c = __popc(__ballot_sync(kFull, below));
        if (c == 32) return hi;
        // probe c is the first at or above q (or past hi): the answer lies
        // after probe c-1 and at or before probe c
        const int pc = lo + step * (c + 1) - 1;
        lo = lo + step * c;
        hi = pc + 1 < hi ? pc + 1 : hi;
    }
    const int pos = lo + lane;
    const bool below = pos < hi && v[pos] < q;
    return lo + __popc(__ballot_sync(kFull, below));
}

// Algorithm 1 for every entry class of a segment, class j in lane j: the same
// machine as fem_machine.cuh's (which keeps all classes in one thread), in
// three registers instead of eighteen, every class stepped by one instruction.
// The last selections of merged classes follow class 0's (their counts are
// kept as offsets from it).
struct Classes {
    int32_t thr, prev;  // this lane's class: threshold, last selection,
    uint32_t cnt;       // count
    // uniform over the warp
    int ncls;
    unsigned live;      // classes not merged into class 0 (bit 0 = class 0)
    int32_t M;
    int open, flags;

    __device__ __forceinline__ void init() {
        thr = prev = 0;
        cnt = 0;
        ncls = 0;
        live = 0;
        M = INT32_MIN;
        open = 1;
        flags = 0;
    }
    // The entry value is known: one class that holds for every value.
    __device__ __forceinline__ void init_known(int32_t x) {
        init();
        thr = INT32_MAX;
        prev = x;
        ncls = 1;
        live = 1u;
        open = 0;
    }
    // An end at t with latest start L (both uniform).
    __device__ __forceinline__ void end(int32_t t, int32_t L, int32_t Tp, int lane) {
        if (((live >> lane) & 1u) && L > prev) {
            cnt += 1;
            prev = t;
        }
        if (open && L > M) {
            if (ncls < kClasses) {
                if (lane == ncls) {
                    thr = L;
                    cnt = 1;
                    prev = t;
                }
                live |= 1u << ncls;
                ncls += 1;
            } else {
                flags |= kMetaClassOverflow;
            }
            M = L;
            if (L >= Tp) open = 0;
        }
        const int32_t prev0 = __shfl_sync(kFull, prev, 0);
        const uint32_t cnt0 = __shfl_sync(kFull, cnt, 0);
        const bool merge = lane > 0 && ((live >> lane) & 1u) && prev == prev0;
        if (merge) cnt -= cnt0;
        live &= ~__ballot_sync(kFull, merge);
    }
    __device__ __forceinline__ void finish(int lane) {
        const int32_t prev0 = __shfl_sync(kFull, prev, 0);
        const uint32_t cnt0 = __shfl_sync(kFull, cnt, 0);
        if (lane > 0 && lane < ncls && !((live >> lane) & 1u)) {
            cnt += cnt0;
            prev = prev0;
        }
    }
    // The segment's record (see write_record), one word per lane.
    __device__ __forceinline__ void write(int32_t *dst, int lane) const {
        const int j = (lane + kClasses - 1) % kClasses;  // the class of word `lane`
        const int32_t a = __shfl_sync(kFull, thr, j), c = __shfl_sync(kFull, prev, j);
        const int32_t b = __shfl_sync(kFull, (int32_t)cnt, j);
        int32_t w = ncls | flags | (open ? 0 : kMetaClosed);
        if (lane > 0) w = lane <= kClasses ? a : lane <= 2 * kClasses ? b : lane <= 3 * kClasses ? c : 0;
        if (lane < kRecWords) dst[lane] = w;
    }
};

// Algorithm 1 over one chunk's valid ends (lane order = time order): the
// steady state jumps from selection to selection, otherwise every end goes
// through every entry class.
__device__ __forceinline__ void greedy_chunk(unsigned bm, int32_t t, int32_t Lv, Classes &st, int32_t Tp, int lane) {
    if (bm && !st.open && st.live == 1u) {
        // the next selection is the first later end whose latest start is
        // after the last selected end
        int32_t prev = __shfl_sync(kFull, st.prev, 0);
        uint32_t added = 0;
        for (;;) {
            const unsigned sel = __ballot_sync(kFull, ((bm >> lane) & 1u) && Lv > prev);
            if (!sel) break;
            const int b = __ffs(sel) - 1;
            prev = __shfl_sync(kFull, t, b);
            ++added;
            bm &= (b == 31) ? 0u : ~((2u << b) - 1u);
        }
        if (lane == 0) {
            st.cnt += added;
            st.prev = prev;
        }
    } else {
        while (bm) {
            const int b = __ffs(bm) - 1;
            bm &= bm - 1;
            st.end(__shfl_sync(kFull, t, b), __shfl_sync(kFull, Lv, b), Tp, lane);
        }
    }
}

// Entries of node k-1 as one step sees them: node 0's are its type's event
// times (latest start = time); later nodes' are (time, latest start) pairs
// in the warp's buffer, so one 8-byte load brings both.  Which of the two is
// known only at run time, uniformly: a copy of every step for either would
// double the kernel's code, and warps at different steps then wait for
// instructions (mixed sizes over 1M events: a third of the stall cycles;
// 9.6 -> 8.6 ms).
struct Entries {
    const void *__restrict__ p;  // node 0's times, or (pairs) a later node's entries
    bool pairs;
    __device__ __forceinline__ int2 get(int i) const {
        if (pairs) return static_cast<const int2 *>(p)[i];
        const int32_t v = static_cast<const int32_t *>(p)[i];
        return make_int2(v, v);
    }
};

// Rank of q among the 32 ascending values v of the warp's lanes: how many are
// below it (0..32).
__device__ __forceinline__ int rank32(int32_t v, int32_t q) {
    const int32_t top = __shfl_sync(kFull, v, 31);
    int c = 0;
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1)
        if (__shfl_sync(kFull, v, c + s - 1) < q) c += s;
    return c == 31 && top < q ? 32 : c;
}

// One node step for one warp: node k's events ev[0, n_ev) (time order)
// against node k-1's entries p[0, m).  An event is valid when the newest
// entry older than t - lo exists and is not older than t - hi; its latest
// start is that entry's.  Not LAST: the valid events are appended to out as
// (t, L) and their number is returned.  LAST: the valid events at or after
// Tp are passed, in time order, to Algorithm 1 of every entry class in st.
//
// Each chunk of 32 events ranks its queries in windows of 32 entries that
// start one entry before the previous chunk's last rank and move on by 31:
// the first entry of every window is older than every query still looking,
// so a lane's predecessor is always in the window where its rank falls and
// its time and latest start are read from the window's registers by a
// shuffle.
template <bool LAST>
__device__ __forceinline__ int node_step(const int32_t *__restrict__ ev, int n_ev, Entries p, int m,
                                         int32_t lo_e, int32_t hi_e, int2 *__restrict__ out, Classes &st,
                                         int32_t Tp, int lane) {
    // All positions fit 32 bits: a recording has fewer than 2^30 events.
    // Times are >= 0 and 0 <= lo < hi, so t - lo and t - hi stay in int32.
    int w = 0;   // entries below the previous chunk's last query
    int wc = 0;  // entries written
    int32_t t_next = lane < n_ev ? ev[lane] : INT32_MAX;
    for (int base = 0; base < n_ev; base += 32) {
        const bool in = base + lane < n_ev;
        const int32_t t = t_next;
        if (base + 32 < n_ev) t_next = (base + 32 + lane < n_ev) ? ev[base + 32 + lane] : INT32_MAX;
        const int32_t q = t - lo_e;
        const int32_t q0 = __shfl_sync(kFull, q, 0);
        int ws = w > 0 ? w - 1 : 0;
        int idx = 0;
        int32_t aT = INT32_MIN, aL = 0;
        bool done = !in;
        for (;;) {
            const int wi = ws + lane;
            const int2 v = wi < m ? p.get(wi) : make_int2(INT32_MAX, 0);
            const int32_t top = __shfl_sync(kFull, v.x, 31);
            if (top < q0 && ws + 32 < m) {  // the whole window precedes every query
                ws += 31;
                continue;
            }
            const int c = rank32(v.x, q);
            const int src = c > 0 ? c - 1 : 0;
            const int32_t xt = __shfl_sync(kFull, v.x, src);
            const int32_t xl = __shfl_sync(kFull, v.y, src);
            if (!done && c < 32) {
                idx = ws + c;
                aT = c > 0 ? xt : INT32_MIN;
                aL = xl;
                done = true;
            }
            if (__all_sync(kFull, done)) break;
            ws += 31;
        }
        const bool ok = in && aT != INT32_MIN && aT >= t - hi_e;
        const int32_t Lv = ok ? aL : 0;
        if (!LAST) {
            const unsigned bm = __ballot_sync(kFull, ok);
            if (ok) out[wc + __popc(bm & ((1u << lane) - 1u))] = make_int2(t, Lv);
            wc += __popc(bm);
        } else {
            greedy_chunk(__ballot_sync(kFull, ok && t >= Tp), t, Lv, st, Tp, lane);
        }
        // the next 32 queries rank at or after this chunk's last one
        w = __shfl_sync(kFull, idx, 31);
    }
    __syncwarp();
    return wc;
}

// Node steps driven by node k-1's entries instead of node k's events, for
// entry lists shorter than the event list.
//
// An event t takes the newest entry i with T_i < t - lo, so the events of
// entry i are those in (T_i + lo, T_{i+1} + lo]; they all carry L_i and are
// valid while t <= T_i + hi.  The intervals of successive entries follow one
// another, so entries in order serve events in time order.
//
// An interval's first event is looked up in the stream's per-type time index:
// the cell of a time gives the list position of the first event at or after
// the cell's start, about one event of the type per cell.
//
// The index row of one type, and the item's part [cb, ce) of its list tl.
struct TypeIndex {
    const int32_t *__restrict__ tl;
    const int32_t *__restrict__ row;  // ncell + 1 cells of 2^shift ticks from tbase
    uint32_t tbase;
    int shift;
    uint32_t ncell;
    int cb, ce;
    __device__ __forceinline__ uint32_t cell(uint32_t q) const {
        return min(q > tbase ? (q - tbase) >> shift : 0u, ncell);
    }
    __device__ __forceinline__ uint32_t time(int pos) const { return pos < ce ? (uint32_t)tl[pos] : 0xFFFFFFFFu; }
    // Position of the part's first event at or after q, by bisection between
    // the first events of q's cell and of the next one (in bursts a cell holds
    // tens of events).
    __device__ __forceinline__ int first(uint32_t q) const {
        const uint32_t c = cell(q);
        int lo = max(row[c], cb), hi = min(row[min(c + 1u, ncell)], ce);
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if ((uint32_t)tl[mid] < q) lo = mid + 1; else hi = mid;
        }
        return lo;
    }
};

// Inner node: every event an entry serves becomes an entry of out; returns
// their number.  Most intervals hold none or one event (compacted by ballot);
// in bursts one of the 32 nearly always holds more, so the first four events
// of every interval are read and compared at once, and placed by a scan
// (counting and writing them one by one took a third of the step).  Wide edges
// behind a rare type give intervals of hundreds of events: the end of one past
// kLongInterval is looked up like its start, and the warp writes it together
// (1M events of 8 types, one of them with 20 events, edges 100k events wide, 16
// episodes: 9.0 ms lane by lane, 7.9 stepped by events, 6.4 so).
//
// Entries thin out node by node (60 types at 20 Hz with bursts, 5 ms edges:
// 25%, 12%, 8% of a type's events), so from the third node on the events are
// several times the entries.
constexpr int kLongInterval = 16;

__device__ __forceinline__ int inner_by_entries(const TypeIndex &ix, Entries p, int m, int32_t lo_e, int32_t hi_e,
                                                int2 *__restrict__ out, int lane) {
    // Times are >= 0 and 0 <= lo < hi < 2^31, so sums of two fit an unsigned
    // 32-bit word.
    const uint32_t lo = (uint32_t)lo_e, hi = (uint32_t)hi_e;
    int wc = 0;  // entries written
    int2 next = lane < m ? p.get(lane) : make_int2(-1, 0);
    for (int base = 0; base < m; base += 32) {
        const int i = base + lane;
        const int2 E = next;
        // the next 32 entries; the first of them ends this chunk's last interval
        next = i + 32 < m ? p.get(i + 32) : make_int2(-1, 0);
        const uint32_t T = (uint32_t)E.x, q = T + lo + 1u;
        uint32_t Tn = __shfl_down_sync(kFull, T, 1);
        const uint32_t T_after = __shfl_sync(kFull, (uint32_t)next.x, 0);
        if (lane == 31) Tn = T_after;
        uint32_t end = T + hi;
        if (i + 1 < m) end = min(end, Tn + lo);
        const int pos = i < m ? ix.first(q) : ix.ce;
        // the interval's first four events, side by side
        uint32_t x[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) x[k] = ix.time(pos + k);
        int n = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) n += i < m && x[k] <= end ? 1 : 0;
        const unsigned bm = __ballot_sync(kFull, n > 0);
        if (!__any_sync(kFull, n > 1)) {
            if (n) out[wc + __popc(bm & ((1u << lane) - 1u))] = make_int2((int32_t)x[0], E.y);
            wc += __popc(bm);
        } else {
            if (n == 4) {
                while (n < kLongInterval && ix.time(pos + n) <= end) ++n;
                if (n == kLongInterval) n = ix.first(end + 1u) - pos;
            }
            int at = n;  // inclusive scan over the lanes
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int y = __shfl_up_sync(kFull, at, d);
                if (lane >= d) at += y;
            }
            int2 *o = out + wc + at - n;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (k < n) o[k] = make_int2((int32_t)x[k], E.y);
            for (int k = 4; k < min(n, kLongInterval); ++k) o[k] = make_int2(ix.tl[pos + k], E.y);
            // the warp writes the rest of the long intervals, one by one
            for (unsigned lg = __ballot_sync(kFull, n > kLongInterval); lg; lg &= lg - 1) {
                const int src = __ffs(lg) - 1;
                const int from = __shfl_sync(kFull, pos, src), len = __shfl_sync(kFull, n, src);
                const int to = wc + __shfl_sync(kFull, at, src) - len;
                const int32_t L = __shfl_sync(kFull, E.y, src);
                for (int k = kLongInterval + lane; k < len; k += 32) out[to + k] = make_int2(ix.tl[from + k], L);
            }
            wc += __shfl_sync(kFull, at, 31);
        }
    }
    __syncwarp();
    return wc;
}

// Last node: the ends are offered to Algorithm 1 of every entry class.  Within
// an entry's interval only the first end at or after Tp can matter: L_i <= T_i
// < t, so once it has been offered every entry class has its last selection
// at or above L_i (it selected this end, or it could not), the largest latest
// start seen is at least L_i, and a later end with the same L_i changes no
// class.  So per entry one lookup finds the first event at or after
// q = max(T_i + lo + 1, Tp), offered when it lies in the entry's interval and
// within its upper bound.  The warp takes 32 x K entries at a time (entry
// base + 32 k + lane in lane k's k-th slot) and issues the K index loads of a
// lane, then its K list loads, side by side.
template <int K>
__device__ __forceinline__ void last_by_entries(const TypeIndex &ix, Entries p, int m, int32_t lo_e, int32_t hi_e,
                                                Classes &st, int32_t Tp, int lane) {
    const uint32_t lo = (uint32_t)lo_e, hi = (uint32_t)hi_e, tp = (uint32_t)Tp;
    for (int base = 0; base < m; base += 32 * K) {
        int2 E[K];
#pragma unroll
        for (int k = 0; k < K; ++k) E[k] = base + 32 * k + lane < m ? p.get(base + 32 * k + lane) : make_int2(-1, 0);
        const int nx = base + 32 * K;
        // the first entry of the next chunk (its time bounds this chunk's
        // last interval)
        const uint32_t T_after = nx < m ? (uint32_t)p.get(nx).x : 0xFFFFFFFFu;
        uint32_t q[K], x[K];
        int pos[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            q[k] = max((uint32_t)E[k].x + lo + 1u, tp);
            pos[k] = base + 32 * k + lane < m ? max(ix.row[ix.cell(q[k])], ix.cb) : ix.ce;
        }
#pragma unroll
        for (int k = 0; k < K; ++k) x[k] = ix.time(pos[k]);
#pragma unroll
        for (int k = 0; k < K; ++k)
            while (x[k] < q[k]) x[k] = ix.time(++pos[k]);
        // (not unrolled: one copy of Algorithm 1; the slots rotate instead)
#pragma unroll 1
        for (int k = 0; k < K; ++k) {
            const int i = base + 32 * k + lane;
            const uint32_t T = (uint32_t)E[0].x;
            // the next entry's time: the next lane's, the next slot's first,
            // or the next chunk's first
            uint32_t Tn = __shfl_down_sync(kFull, T, 1);
            const uint32_t Tf = k + 1 < K ? __shfl_sync(kFull, (uint32_t)E[K > 1 ? 1 : 0].x, 0) : T_after;
            if (lane == 31) Tn = Tf;
            // x = the first event at or after q (none: past the item's part)
            const bool ok = i < m && x[0] <= T + hi && (i + 1 >= m || x[0] <= Tn + lo);
            greedy_chunk(__ballot_sync(kFull, ok), (int32_t)x[0], ok ? E[0].y : 0, st, Tp, lane);
#pragma unroll
            for (int j = 0; j + 1 < K; ++j) {
                E[j] = E[j + 1];
                x[j] = x[j + 1];
            }
        }
    }
    __syncwarp();
}

// A work item is one segment p of one recording for either one episode
// (slot) or, with groups, a run of episode slots [s0, s1) that share their
// first N-1 nodes and edges (or, with a.pair, their first two nodes and the
// edge between them, whatever follows): the shared prefix is tracked once, and
// only the remaining node steps are run per episode.
__global__ void __launch_bounds__(kTrackWarps * 32, kTrackMaxBlocksPerSm) k_count_track(TrackArgs a) {
    const int lane = threadIdx.x & 31;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    // entry lists of (time, latest start) pairs: two used in turn, or, where
    // the slots of a group share their first two nodes, that prefix's list
    // and two more
    int2 *const b0 = reinterpret_cast<int2 *>(a.buf + gw * (a.pair ? 6 : 4) * a.cap);
    const int64_t n_items = a.d_n_items ? *a.d_n_items : a.n_items;
    for (;;) {
        unsigned long long it = 0;
        if (lane == 0) it = atomicAdd(a.queue, 1ull);
        it = __shfl_sync(kFull, it, 0);
        if ((int64_t)it >= n_items) break;
        int r = 0, P = 1, p = 0, s0 = 0, s1 = 0;
        if (a.ibase) {
            // items numbered recording by recording in the order rorder
            // (longest recordings first), each recording's groups (or
            // slots) times its segments
            int lo_r = 0, hi_r = a.n_recs;  // last position whose items start at or before it
            while (hi_r - lo_r > 1) {
                const int mid = (lo_r + hi_r) >> 1;
                if (a.ibase[mid] <= (int64_t)it) lo_r = mid; else hi_r = mid;
            }
            r = a.rorder ? a.rorder[lo_r] : lo_r;
            P = a.rinfo[r].P;
            const int64_t local = (int64_t)it - a.ibase[lo_r];
            const int64_t g = a.gfirst[r] + local / P;
            p = (int)(local % P);
            if (a.gstart) {
                s0 = a.gstart[g];
                s1 = a.gstart[g + 1];
            } else {
                s0 = (int)g;
                s1 = s0 + 1;
            }
        } else {
            const int64_t tr = a.rec_first + (int64_t)it;
            int lo_r = 0, hi_r = a.n_recs;  // last recording whose records start at or before tr
            while (hi_r - lo_r > 1) {
                const int mid = (lo_r + hi_r) >> 1;
                if (a.rinfo[mid].recbase <= tr) lo_r = mid; else hi_r = mid;
            }
            r = lo_r;
            P = a.rinfo[r].P;
            const int64_t local = tr - a.rinfo[r].recbase;
            s0 = a.rinfo[r].slot_first + (int)(local / P);
            s1 = s0 + 1;
            p = (int)(local % P);
        }
        const RecInfo &ri = a.rinfo[r];
        // halo: the largest sum of upper bounds over the item's episodes (one
        // per lane; a sum past INT32_MAX reaches back before every event);
        // no work when a bound dropped every episode of the item
        uint32_t hsum = 0;
        bool kept = false;
        for (int s = s0 + lane; s < s1; s += 32) {
            const int c = a.slot2cand[s];
            const int64_t o = a.offs[c], e = a.offs[c + 1];
            int64_t h = 0;
            for (int64_t k = o - c; k < e - c - 1; ++k) h += a.chi[k];
            hsum = max(hsum, (uint32_t)min(h, (int64_t)INT32_MAX));
            kept = kept || (e - o >= 2 && !(a.skip && a.skip[c]));
        }
        const uint32_t sumhi = __reduce_max_sync(kFull, hsum);
        const int64_t seg_b = ri.seg[p], seg_e = ri.seg[p + 1];
        const bool live = seg_b < seg_e && __any_sync(kFull, kept);
        int32_t Tp = 0, haloT = 0, Tend = INT32_MAX;  // (times are below INT32_MAX)
        if (live) {
            Tp = ri.time[seg_b];
            haloT = Tp - (int32_t)sumhi;
            if (seg_e < ri.n) Tend = ri.time[seg_e];
        }
        // list range of type E inside [haloT, Tend)
        auto range = [&](uint32_t E, int &b, int &e) {
            const int b0 = (int)ri.toff[E], b1 = (int)ri.toff[E + 1];
            if (ri.tseg) {
                const int32_t *tq = ri.tseg + (size_t)E * ri.tstride;
                const int qmax = ri.tstride - 1;
                const int st0 = b0 + tq[min(p * ri.sstep, qmax)];
                e = b0 + tq[min((p + 1) * ri.sstep, qmax)];
                b = (p == 0) ? st0 : warp_lower_bound(ri.ttime, b0, st0, haloT, lane);
            } else {
                b = (p == 0) ? b0 : warp_lower_bound(ri.ttime, b0, b1, haloT, lane);
                e = Tend != INT32_MAX ? warp_lower_bound(ri.ttime, b, b1, Tend, lane) : b1;
            }
        };
        // whether a node with n_ev events is stepped by node k-1's m entries:
        // the entry steps' scattered lookups cost about two streamed events
        // (the same 200k episodes: 143 ms with the line at 1, 131 at 2, 130 at
        // 3; 48 recordings with groups of 3-node episodes are fastest at 1-2)
        auto by_entries = [&](int m, int n_ev) {
            return ri.tidx &&
                   (a.last_mode == 2 || (a.last_mode == 0 && (int64_t)m * kTrackEntryRatio < (int64_t)n_ev));
        };
        auto index_of = [&](uint32_t E, int cb, int ce) {
            const int t0 = (int)ri.toff[E];
            return TypeIndex{ri.ttime + t0, ri.tidx + (int64_t)E * (ri.tcells + 1), (uint32_t)ri.tbase, ri.tshift,
                             (uint32_t)ri.tcells, cb - t0, ce - t0};
        };
        // Every episode of the item: node 0 (its type's times), nodes 1..N-2
        // (entry lists in the warp's buffer), the last node.  The first one
        // tracks the prefix that the item's episodes share, whose last list
        // (node `depth`, m_pre entries) the others start from.
        Entries en{nullptr, false};
        int m_pre = 0;
        bool tracked = false;
        Classes st;
        for (int s = s0; s < s1; ++s) {
            const int c = a.slot2cand[s];
            const bool direct = P == 1 && a.counts;
            if (a.skip && a.skip[c]) {  // pruned by a bound: count 0 (else the stitch writes it)
                if (direct && lane == 0) a.counts[c] = 0;
                continue;
            }
            const int64_t oc = a.offs[c], ec = oc - c;
            const int N = (int)(a.offs[c + 1] - oc);
            const int depth = a.pair ? 1 : N - 2;
            int m = 0;
            if (live && N >= 2) {
                int k = depth + 1;
                if (!tracked) {
                    tracked = true;
                    int b = 0, e = 0;
                    range(a.ctypes[oc], b, e);
                    en.p = ri.ttime + b;
                    en.pairs = false;
                    m = e - b;
                    k = 1;
                    if (depth == 0) m_pre = m;
                } else {
                    m = m_pre;
                    en.p = b0 + a.cap * (depth & 1);
                    en.pairs = true;
                }
                for (; k < N - 1 && m > 0; ++k) {
                    int cb = 0, ce = 0;
                    range(a.ctypes[oc + k], cb, ce);
                    // the list after the next one, sparing the shared prefix's
                    int2 *out = b0 + a.cap * ((k & 1) ? (a.pair && k > 1 ? 2 : 1) : 0);
                    const int32_t lo_k = a.relaxed ? 0 : a.clo[ec + k - 1], hi_k = a.chi[ec + k - 1];
                    if (by_entries(m, ce - cb)) {
                        m = inner_by_entries(index_of(a.ctypes[oc + k], cb, ce), en, m, lo_k, hi_k, out, lane);
                    } else {
                        m = node_step<false>(ri.ttime + cb, ce - cb, en, m, lo_k, hi_k, out, st, 0, lane);
                    }
                    en.p = out;
                    en.pairs = true;
                    if (k == depth) m_pre = m;
                }
            }
            const bool known = a.prev && p == 0;
            if (known) st.init_known(a.prev[c]); else st.init();
            if (m > 0) {
                int cb = 0, ce = 0;
                range(a.ctypes[oc + N - 1], cb, ce);
                // appended events: the retained tail's ends were offered before
                if (known) {
                    const uint32_t E = a.ctypes[oc + N - 1];
                    cb = min(ce, max(cb, (int)ri.toff[E] + a.tail_cnt[E]));
                }
                const int n_ev = ce - cb;
                const int32_t lo_l = a.relaxed ? 0 : a.clo[ec + N - 2], hi_l = a.chi[ec + N - 2];
                if (by_entries(m, n_ev)) {
                    last_by_entries<kTrackEntrySlots>(index_of(a.ctypes[oc + N - 1], cb, ce), en, m, lo_l, hi_l, st,
                                                      Tp, lane);
                } else {
                    node_step<true>(ri.ttime + cb, n_ev, en, m, lo_l, hi_l, nullptr, st, Tp, lane);
                }
            }
            st.finish(lane);
            if (!direct)
                st.write(a.rec + (ri.recbase + (int64_t)(s - ri.slot_first) * P + p) * kRecWords, lane);
            else if (lane == 0)
                // one segment from the recording's start: the first valid
                // end closes the entry classes at class 0, whose count is
                // the episode's (what the stitch would read)
                a.counts[c] = st.ncls > 0 ? st.cnt : 0u;
        }
    }
}

// Groups for the grouped launch: flag[s] = 1 where slot s starts a group
// (first slot, another recording or size, a different prefix of N-1 nodes
// and N-2 edges, or every kTrackGroupMax-th slot; with `pair` sizes may differ
// and the prefix is two nodes and one edge).  Episodes of one to two
// nodes share nothing and stay alone.
__global__ void k_track_group_flags(const int32_t *__restrict__ slot2cand, const int32_t *__restrict__ d_n_slots,
                                    int64_t n_slots_cap, const int64_t *__restrict__ offs,
                                    const uint16_t *__restrict__ ctypes, const int32_t *__restrict__ clo,
                                    const int32_t *__restrict__ chi, const uint32_t *__restrict__ cand_rec,
                                    int pair, int32_t *__restrict__ flag) {
    const int64_t n = d_n_slots ? (int64_t)*d_n_slots : n_slots_cap;
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s <= n_slots_cap;
         s += (int64_t)gridDim.x * blockDim.x) {
        if (s >= n) {
            flag[s] = 0;
            continue;
        }
        bool f = (s == 0) || (s % (pair ? kTrackPairMax : kTrackGroupMax)) == 0;
        if (!f) {
            const int c = slot2cand[s], b = slot2cand[s - 1];
            const int64_t oc = offs[c], ob = offs[b];
            const int N = (int)(offs[c + 1] - oc), Nb = (int)(offs[b + 1] - ob);
            f = (pair ? Nb < 3 : N != Nb) || N < 3 || (cand_rec && cand_rec[c] != cand_rec[b]);
            const int sh = pair ? 2 : N - 1;  // shared nodes
            for (int k = 0; k < sh && !f; ++k) f = ctypes[oc + k] != ctypes[ob + k];
            for (int k = 0; k < sh - 1 && !f; ++k)
                f = clo[oc - c + k] != clo[ob - b + k] || chi[oc - c + k] != chi[ob - b + k];
        }
        flag[s] = f ? 1 : 0;
    }
}

// After an exclusive scan of the flags in place (gidx[s] = groups before
// slot s, gidx[n] = all groups): the first slot of every group, and (one
// thread) per recording its first group and its first item (groups x
// segments), and the item count.
__global__ void k_track_group_starts(const int32_t *__restrict__ gidx, const int32_t *__restrict__ d_n_slots,
                                     int64_t n_slots_cap, int32_t *__restrict__ gstart,
                                     const int32_t *__restrict__ slot2cand, const uint32_t *__restrict__ cand_rec,
                                     int32_t *__restrict__ gmax) {
    const int64_t n = d_n_slots ? (int64_t)*d_n_slots : n_slots_cap;
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s <= n; s += (int64_t)gridDim.x * blockDim.x) {
        if (s == n) {
            gstart[gidx[n]] = (int32_t)n;
        } else if (gidx[s + 1] != gidx[s]) {
            gstart[gidx[s]] = (int32_t)s;
            if (gmax) {
                // the group runs to the next start (at most kTrackGroupMax slots)
                int64_t j = s + 1;
                while (j < n && gidx[j + 1] == gidx[j]) ++j;
                atomicMax(gmax + (cand_rec ? cand_rec[slot2cand[s]] : 0u), (int32_t)(j - s));
            }
        }
    }
}

// Per recording (one thread): its first group (or, without groups, its first
// slot) and, walking the recordings in the order rorder, the first item of
// each (groups x segments) and the item count.
__global__ void k_track_group_recs(const int32_t *__restrict__ gidx, const RecInfo *__restrict__ rinfo, int n_recs,
                                   const int32_t *__restrict__ rorder, const int32_t *__restrict__ d_n_slots,
                                   int64_t n_slots_cap, int32_t *__restrict__ gfirst, int64_t *__restrict__ ibase,
                                   int64_t *n_items) {
    const int64_t n = d_n_slots ? (int64_t)*d_n_slots : n_slots_cap;
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    auto first = [&](int r) -> int64_t {
        const int64_t sf = r < n_recs ? (int64_t)rinfo[r].slot_first : n;
        const int64_t c = sf < n ? sf : n;
        return gidx ? (int64_t)gidx[c] : c;
    };
    int64_t base = 0;
    for (int i = 0; i < n_recs; ++i) {
        const int r = rorder ? rorder[i] : i;
        const int64_t g0 = first(r), g1 = first(r + 1);
        gfirst[r] = (int32_t)g0;
        ibase[i] = base;
        base += (g1 - g0) * rinfo[r].P;
    }
    ibase[n_recs] = base;
    *n_items = base;
}

}  // namespace

// Sort keys of slots for groups by the first two nodes: 0 = the first edge
// (its bounds hashed to kPairEdgeKeys values: unequal edges with one key only
// cut a group), 1 = the second node, 2 = the first node, 3 = the recording.
__global__ void k_track_pair_keys(const int32_t *__restrict__ slot2cand, int64_t n, const int64_t *__restrict__ offs,
                                  const uint16_t *__restrict__ ctypes, const int32_t *__restrict__ clo,
                                  const int32_t *__restrict__ chi, const uint32_t *__restrict__ cand_rec, int which,
                                  int32_t *__restrict__ key) {
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
        const int c = slot2cand[s];
        const int64_t o = offs[c];
        int32_t k = 0;
        if (which == 3)
            k = cand_rec ? (int32_t)cand_rec[c] : 0;
        else if (which == 2)
            k = ctypes[o];
        else if (which == 1)
            k = offs[c + 1] - o >= 2 ? (int32_t)ctypes[o + 1] : 0;
        else if (offs[c + 1] - o >= 3)
            // (episodes that share nothing come first, so that they cut no group)
            k = 1 + (int32_t)((((uint32_t)clo[o - c] * 2654435761u) ^ ((uint32_t)chi[o - c] * 2246822519u)) >> 8) %
                        (kPairEdgeKeys - 1);
        key[s] = k;
    }
}

int track_group_flags(cudaStream_t st, int n_sm, const TrackGroupIn &in) {
    const int64_t cap = in.n_slots_cap;
    const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>((cap + 256) / 256, 8 * (int64_t)n_sm));
    k_track_group_flags<<<g, 256, 0, st>>>(in.slot2cand, in.d_n_slots, cap, in.offs, in.ctypes, in.clo, in.chi,
                                           in.cand_rec, in.pair ? 1 : 0, in.gidx);
    FEM_CUDA_TRY(cudaGetLastError());
    return FEM_OK;
}

int track_group_starts(cudaStream_t st, int n_sm, const TrackGroupIn &in) {
    const int64_t cap = in.n_slots_cap;
    const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>((cap + 256) / 256, 8 * (int64_t)n_sm));
    FEM_TRY(track_group_flags(st, n_sm, in));
    FEM_TRY(scan_exclusive(st, in.gidx, cap + 1, in.scan_tmp, nullptr, nullptr));
    if (in.gmax && cudaMemsetAsync(in.gmax, 0, sizeof(int32_t) * std::max(in.n_recs, 1), st) != cudaSuccess)
        return FEM_ERR_CUDA;
    k_track_group_starts<<<g, 256, 0, st>>>(in.gidx, in.d_n_slots, cap, in.gstart, in.slot2cand, in.cand_rec,
                                            in.gmax);
    FEM_CUDA_TRY(cudaGetLastError());
    return FEM_OK;
}

void track_pair_keys(cudaStream_t st, int n_sm, const TrackGroupIn &in, int which, int32_t *key) {
    const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>((in.n_slots_cap + 255) / 256, 8 * (int64_t)n_sm));
    k_track_pair_keys<<<g, 256, 0, st>>>(in.slot2cand, in.n_slots_cap, in.offs, in.ctypes, in.clo, in.chi,
                                         in.cand_rec, which, key);
}

int track_groups(cudaStream_t st, int n_sm, const TrackGroupIn &in, bool grouped, TrackArgs *a) {
    const int64_t cap = in.n_slots_cap;
    if (grouped && !in.starts_ready) FEM_TRY(track_group_starts(st, n_sm, in));
    k_track_group_recs<<<1, 32, 0, st>>>(grouped ? in.gidx : nullptr, in.rinfo, in.n_recs, in.rorder, in.d_n_slots,
                                         cap, in.gfirst, in.ibase, in.n_items);
    FEM_CUDA_TRY(cudaGetLastError());
    a->pair = grouped && in.pair ? 1 : 0;
    a->gstart = grouped ? in.gstart : nullptr;
    a->gfirst = in.gfirst;
    a->ibase = in.ibase;
    a->rorder = in.rorder;
    a->d_n_items = in.n_items;
    return FEM_OK;
}

int track_blocks(int n_sm) {
    int per_sm = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_count_track, kTrackWarps * 32, 0);
    cudaGetLastError();
    return std::max(1, n_sm) * std::max(1, std::min(per_sm, kTrackMaxBlocksPerSm));
}

size_t track_buf_bytes(int blocks, int64_t cap, bool pair) {
    return (size_t)blocks * kTrackWarps * (pair ? 6 : 4) * (size_t)std::max<int64_t>(cap, 1) * sizeof(int32_t);
}

int launch_track(cudaStream_t st, int blocks, const TrackArgs &a, bool reset) {
    if (blocks < 1) return FEM_OK;
    if (reset && cudaMemsetAsync(a.queue, 0, sizeof(unsigned long long), st) != cudaSuccess) return FEM_ERR_CUDA;
    k_count_track<<<(unsigned)blocks, kTrackWarps * 32, 0, st>>>(a);
    FEM_CUDA_TRY(cudaGetLastError());
    return FEM_OK;
}

}  // namespace fem
