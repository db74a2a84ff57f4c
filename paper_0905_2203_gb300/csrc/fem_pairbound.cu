// fem_pairbound.cu -- upper bound on the count of every 2-node episode of a
// recording in one pass over its events (anti-monotonicity, section
// "Temporal Data Mining").
//
// The non-overlapped occurrences of a -(lo, hi]-> b end at distinct b-events,
// each with an a-event inside its window, so
//     count(a, b, bin) <= UB = #{ b-events with an a-event in the window }.
// Event i of type a, with the type's next event gap ticks later, is the
// newest a-event of j's window (t_j - hi, t_j - lo] exactly when
//     lo < t_j - t_i <= min(hi, lo + gap),
// so every (a-event, bin) pair adds one to UB(a, type_j, bin) for each event
// j of that range and no b-event is counted twice.
//
// What bounds it: one update per (event, event of its look-ahead window), 20
// to 130 per event.  A thread per event that looks back and adds to the table
// in global memory makes each of them a scattered L2 reduction (20M events of
// 256 types at 25 Hz, 2.6e9 updates: 14.7 ms, 1.7e11 updates/s).  Here a block
// takes a run of ONE type's event list, so all its updates fall into the
// type's row of the table (n_types x bins counters), which it keeps in shared
// memory and adds to the global table once; eight lanes take one event and
// read the events after it side by side, so the loads are coalesced and no
// per-thread bitset is needed.  Mining calls by this kernel, with 32 lanes an
// event from 12 events on, and by the look-back: 20M events from host memory
// (128 events a window) 6.1, 7.1 and 29.5 ms; 1.07M events of 128 types (21
// events) 536, 560 and 870 us.  At 36 registers (6 blocks per SM) it issues on
// 67% of the cycles over the latter.
#include <algorithm>

#include "fem_internal.cuh"

namespace fem {

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr int kPbThreads = 256;
constexpr int kPbLanes = 8;                  // lanes of an event ...
constexpr unsigned kPbLasts = 0x80808080u;   // ... and the last lane of each group
constexpr int kPbWarps = kPbThreads / 32;
constexpr int kPbMinChunk = 256, kPbMaxChunk = 4096;  // list positions per block

// A warp's share of a chunk, at most its lanes and a multiple of the events it
// takes side by side.
__host__ __device__ constexpr int pair_bound_batch(int chunk) {
    const int b = chunk / kPbWarps;
    return b >= 32 ? 32 : b <= 32 / kPbLanes ? 32 / kPbLanes : b / (32 / kPbLanes) * (32 / kPbLanes);
}

// Which bin a distance falls into.  NB = 0: nb adjacent bins of one width (the
// usual case), found by one multiplication; the newest-event condition is
// then rem < min(width, gap) whatever the bin.  NB > 0: any bins, up to NB of
// them, each tested (they may overlap or leave gaps).
template <int NB>
struct Bins {
    int32_t lo[NB];
    uint32_t width[NB], len[NB];
    __device__ __forceinline__ explicit Bins(const PairBoundArgs &a) {
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            lo[k] = k < a.nb ? a.blo[k] : 0;
            width[k] = k < a.nb ? (uint32_t)(a.bhi[k] - a.blo[k]) : 0u;  // 0: no such bin
        }
    }
    __device__ __forceinline__ void event(uint32_t gap) {
#pragma unroll
        for (int k = 0; k < NB; ++k) len[k] = min(width[k], gap);
    }
    __device__ __forceinline__ void add(uint32_t *h, int32_t d, int nt) const {
#pragma unroll
        for (int k = 0; k < NB; ++k)
            if ((uint32_t)(d - lo[k] - 1) < len[k]) atomicAdd(h + k * nt, 1u);
    }
};
template <>
struct Bins<0> {
    int32_t first;  // lower bound of the first bin, plus one
    uint32_t nb, width, magic, len;
    __device__ __forceinline__ explicit Bins(const PairBoundArgs &a)
        : first(a.blo[0] + 1), nb((uint32_t)a.nb), width(a.width), magic(a.magic) {}
    __device__ __forceinline__ void event(uint32_t gap) { len = min(width, gap); }
    // x: distance past the first bin's lower bound (as unsigned, far above
    // every bin when it is short of it); all = nb * width
    __device__ __forceinline__ void add(uint32_t *row, int32_t x, uint32_t b, int nt, int32_t all) const {
        const uint32_t k = __umulhi((uint32_t)x, magic);  // x / width for x < all
        const bool ok = (uint32_t)x < (uint32_t)all && (uint32_t)x - k * width < len;
        if (ok) atomicAdd(row + (k * (uint32_t)nt + b), 1u);
    }
};

template <int NB>
__global__ void __launch_bounds__(kPbThreads, NB == 0 ? 6 : 4) k_pair_bound(PairBoundArgs a) {
    constexpr int G = kPbLanes;
    extern __shared__ uint32_t s_row[];  // counter of (bin k, type b) at k * nt + b: neighbouring types, other banks
    constexpr int kSide = 32 / G;        // events a warp takes side by side
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int batch = pair_bound_batch(a.chunk);  // list positions a warp takes at a time
    Bins<NB> bins(a);
    const int32_t all = a.nb * (int32_t)a.width;  // (NB = 0) the windows' whole width
    for (int64_t item = blockIdx.x; item < a.n_items; item += gridDim.x) {
        int r = 0;
        for (int hi_r = a.n_recs; hi_r - r > 1;) {
            const int mid = (r + hi_r) >> 1;
            if (a.cpre[mid] <= item) r = mid; else hi_r = mid;
        }
        const RecInfo &ri = a.ri[r];
        const int n = (int)ri.n;
        const int32_t *__restrict__ tm = ri.time;
        const uint16_t *__restrict__ ty = ri.type;
        const int32_t *__restrict__ tl = ri.ttime;
        const int32_t *__restrict__ tp = ri.tpos;
        const int nt = (int)a.nt[r], words = nt * a.nb;
        const int c0 = (int)((item - a.cpre[r]) * a.chunk), c1 = min(n, c0 + a.chunk);
        int E = 0;  // type of list position c0: toff[E] <= c0 < toff[E + 1]
        for (int hi_e = nt; hi_e - E > 1;) {
            const int mid = (E + hi_e) >> 1;
            if (ri.toff[mid] <= c0) E = mid; else hi_e = mid;
        }
        for (int p = c0; p < c1; ++E) {
            const int te = (int)ri.toff[E + 1];  // end of the type's list
            const int p1 = min(c1, te);
            if (p1 <= p) continue;
            // an infrequent type is in no level-2 candidate
            if (ri.freq[E] > a.thr[r]) {
                for (int w = threadIdx.x; w < words; w += kPbThreads) s_row[w] = 0;
                __syncthreads();
                for (int base = p + warp * batch; base < p1; base += kPbWarps * batch) {
                    const int q = base + lane;
                    const int32_t t = q < p1 ? tl[q] : 0;
                    const int32_t at = q < p1 ? tp[q] : 0;
                    const uint32_t gap = q < p1 && q + 1 < te ? (uint32_t)(tl[q + 1] - t) : 0xFFFFFFFFu;
                    const int cnt = min(batch, p1 - base);
                    for (int e = 0; e < cnt; e += kSide) {
                        const int src = e + lane / G;  // below 32: e is a multiple of kSide
                        const int32_t ti = __shfl_sync(kFull, t, src);
                        bins.event(__shfl_sync(kFull, gap, src));
                        int j = __shfl_sync(kFull, at, src) + 1 + (lane & (G - 1));
                        if (src >= cnt) j = n;
                        if constexpr (NB == 0) {
                            // Past the last event the stream is padded with
                            // times no window reaches (checked on the host),
                            // for more events than a warp runs past the end;
                            // the next G events are loaded before these are
                            // used.  A group goes on while its last lane is
                            // inside the window.
                            const int32_t base_t = ti + bins.first;
                            const int32_t *pt = tm + j;
                            const uint16_t *py = ty + j;
                            int32_t tj = *pt;
                            uint32_t b = *py;
                            for (;;) {
                                const int32_t x = tj - base_t;
                                const uint32_t bj = b;
                                pt += G;
                                py += G;
                                tj = *pt;
                                b = *py;
                                bins.add(s_row, x, bj, nt, all);
                                const unsigned bm = __ballot_sync(kFull, x < all);
                                if (!(bm & kPbLasts)) break;
                                // a finished group waits at the padding
                                if (!((bm >> (lane | (G - 1))) & 1u)) {
                                    pt = tm + n;
                                    py = ty + n;
                                    tj = INT32_MAX;
                                }
                            }
                        } else {
                            for (;; j += G) {
                                const bool in = j < n;
                                const int32_t d = (in ? tm[j] : 0) - ti;
                                const uint32_t b = in ? ty[j] : 0;
                                const bool win = in && d <= a.hi_max;
                                if (win) bins.add(s_row + b, d, nt);
                                const unsigned bm = __ballot_sync(kFull, win);
                                if (!((bm >> (lane | (G - 1))) & 1u)) j = n;
                                if (!__any_sync(kFull, j < n)) break;
                            }
                        }
                    }
                }
                __syncthreads();
                uint32_t *u = a.ub + a.ub_off[r] + (size_t)E * words;
                for (int w = threadIdx.x; w < words; w += kPbThreads) {
                    const uint32_t v = s_row[w];
                    if (v) atomicAdd(u + (w % nt) * a.nb + w / nt, v);
                }
                __syncthreads();
            }
            p = p1;
        }
    }
}

}  // namespace

// Chunk length (list positions per block): about four blocks per resident
// one over all recordings, so that the last wave is short, between 256 (a
// batch of 32 events per warp) and 4096 (the row's flush is then under 1% of
// the updates).  Fewer events than fill the resident blocks that way are dealt
// out over them, down to 4 events per warp: with chunks of 256, 5000 events of
// 500 types (eight uneven bins, 50 events in their windows) make 20 blocks of
// 25 rows each: the whole mining call takes 402 us, 163 with chunks of 32.
int pair_bound_chunk(int n_sm, int64_t events) {
    const int64_t resident = (int64_t)n_sm * 8;
    if (events < resident * kPbMinChunk) {
        const int64_t c = (events / resident + 31) / 32 * 32;
        return (int)std::max<int64_t>(32, std::min<int64_t>(kPbMinChunk, c));
    }
    const int64_t c = events / (resident * 4);
    return (int)std::max<int64_t>(kPbMinChunk, std::min<int64_t>(kPbMaxChunk, (c + 255) / 256 * 256));
}

// blo / bhi: the bins on the host; t_last: the last event time of any
// recording.
int pair_bound(cudaStream_t st, int n_sm, PairBoundArgs a, const std::vector<int32_t> &blo,
               const std::vector<int32_t> &bhi, uint32_t nt_max, int64_t t_last) {
    if (a.n_items < 1) return FEM_OK;
    // adjacent bins of one width; with m = ceil(2^32 / w) the high word of
    // x * m is x / w exactly while x * (m * w - 2^32) < 2^32, so for every
    // x < 8 w when 8 w^2 < 2^32
    const int64_t w = (int64_t)bhi[0] - blo[0];
    bool even = w >= 2 && 8 * w * w < ((int64_t)1 << 32);
    for (int k = 1; k < a.nb; ++k) even = even && blo[k] == bhi[k - 1] && bhi[k] - blo[k] == w;
    even = even && t_last + a.hi_max < INT32_MAX;  // the padding's times lie past every window
    a.width = (uint32_t)w;
    a.magic = even ? (uint32_t)((((uint64_t)1 << 32) + w - 1) / w) : 0u;
    const size_t sm = sizeof(uint32_t) * (size_t)nt_max * (size_t)a.nb;  // at most 1024 x 8 words
    const unsigned grid = (unsigned)std::min<int64_t>(a.n_items, (int64_t)n_sm * 64);
    if (even)
        k_pair_bound<0><<<grid, kPbThreads, sm, st>>>(a);
    else if (a.nb <= 4)
        k_pair_bound<4><<<grid, kPbThreads, sm, st>>>(a);
    else
        k_pair_bound<8><<<grid, kPbThreads, sm, st>>>(a);
    FEM_CUDA_TRY(cudaGetLastError());
    return FEM_OK;
}

}  // namespace fem
