// fem_joinbound.cu -- an upper bound on the count of every 3-node candidate
// from its two frequent 2-node sub-episodes, taken before the exact count.
//
// A level-3 candidate A -(b1]-> B -(b2]-> C is the join of the frequent
// 2-node episodes alpha = A -(b1]-> B and beta = B -(b2]-> C.  Every
// occurrence of the candidate passes through one B event that has an A event
// inside b1 before it (the B event is a valid end of alpha) and a C event
// inside b2 after it (a valid start of beta), and non-overlapped occurrences
// pass through distinct B events.  So
//     count <= UB = #{ B events that are both },
// the same anti-monotonicity argument ("Temporal Data Mining") as the
// level-2 pair bound.  Every frequent 2-node episode X -(b]-> Y of a
// recording gets two bitsets, one bit per event of a type's list: V over
// Y's list (valid ends) and S over X's list (valid starts), each word one
// ballot of a warp over 32 consecutive events, found with the stream's
// per-type time index.  A candidate's UB is then the popcount of
// V(alpha) AND S(beta), both over B's list: about n_B / 32 word operations,
// where its exact count looks at every entry of alpha.  Candidates whose UB
// is at or below the recording's threshold are skipped by the exact count
// (their count is reported as 0 and they cannot be frequent).
//
// Bitsets are laid out per recording: recording r's frequent 2-node
// episodes f (in their order) take stride[r] words each (the longest list of
// the recording / 32), from base[r]; the pass is skipped (nothing pruned)
// when the total passes the buffers' capacity.
#include "fem_internal.cuh"

namespace fem {

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

__device__ __forceinline__ int bin_of(const JoinBoundArgs &a, int32_t lo, int32_t hi) {
    int k = 0;
    while (k < a.nb && !(a.blo[k] == lo && a.bhi[k] == hi)) ++k;
    return k;
}

// List position of the first event at or after the start of q's cell (type
// row `row` of the time index).
__device__ __forceinline__ int cell_of(const RecInfo &ri, const int32_t *__restrict__ row, uint32_t q) {
    const uint32_t tb = (uint32_t)ri.tbase;
    const uint32_t c = q > tb ? (q - tb) >> ri.tshift : 0u;
    return row[min(c, (uint32_t)ri.tcells)];
}

// The (X, Y, bin) -> frequent 2-node episode table (entries set to -1
// before): the episode's index in the frequent set.
__global__ void k_jb_index(JoinBoundArgs a) {
    const int64_t F = *a.f2n;
    for (int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; f < F; f += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t r = a.f2rec[f];
        const int k = bin_of(a, a.f2lo[f], a.f2hi[f]);
        if (k >= a.nb) continue;
        const uint32_t X = a.f2types[2 * f], Y = a.f2types[2 * f + 1];
        a.tab[a.tab_off[r] + ((int64_t)X * a.nt[r] + Y) * a.nb + k] = (int32_t)f;
    }
}

// One thread: the first word of every recording's bitsets and the total.
__global__ void k_jb_base(JoinBoundArgs a) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    int64_t acc = 0;
    for (int r = 0; r < a.n_recs; ++r) {
        a.base[r] = acc;
        acc += (a.f2foff[r + 1] - a.f2foff[r]) * (int64_t)a.stride[r];
    }
    a.base[a.n_recs] = acc;
}

// The V and S bitsets of every frequent 2-node episode.  One warp per (ordered
// pair of types, chunk of list events), for all the pair's frequent bins at
// once: an event of one list looks up the other list's first event inside the
// widest window and walks on to its end, marking the bin of every event it
// meets (0.2 events on average at 12 Hz and 20 ms); then one ballot per bin and
// 32 events.  The lookups are scattered reads, 32 lines each, which is what
// bounds this, and they are made once, not once per bin.  The pair's item is
// that of its first frequent bin.  64 recordings of 60 types (55M events, four
// bins): 12 ms bin by bin, 8 ms so; one 1.07M-event recording 72 -> 51 us, with
// chunks of a 64th of the longest list (2048 events: 212 us, too few items).
// NB: bins held in registers (0: in shared memory, up to 32).
template <int NB>
__global__ void __launch_bounds__(256, 6) k_jb_bits(JoinBoundArgs a) {
    __shared__ int32_t s_lo[kJoinBoundMaxBins], s_hi[kJoinBoundMaxBins];
    if (threadIdx.x < (unsigned)a.nb) {
        s_lo[threadIdx.x] = a.blo[threadIdx.x];
        s_hi[threadIdx.x] = a.bhi[threadIdx.x];
    }
    __syncthreads();
    if (a.base[a.n_recs] > a.cap_words) return;
    const int lane = threadIdx.x & 31;
    const int64_t items = (int64_t)*a.f2n * a.nch;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t it = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; it < items; it += nw) {
        const int64_t f = it / a.nch;
        const int b0 = (int)(it - f * a.nch) * a.chunk, b1 = b0 + a.chunk;
        const uint32_t r = a.f2rec[f];
        const RecInfo &ri = a.ri[r];
        const uint32_t X = a.f2types[2 * f], Y = a.f2types[2 * f + 1];
        const int64_t xb = ri.toff[X], yb = ri.toff[Y];
        const int lenX = (int)(ri.toff[X + 1] - xb), lenY = (int)(ri.toff[Y + 1] - yb);
        if (b0 >= lenX && b0 >= lenY) continue;
        // the pair's frequent bins: lane k holds bin k's episode (-1: none)
        const int32_t *tab = a.tab + a.tab_off[r] + ((int64_t)X * a.nt[r] + Y) * a.nb;
        const int32_t fk = lane < a.nb ? tab[lane] : -1;
        const unsigned bins = __ballot_sync(kFull, fk >= 0);
        if (__shfl_sync(kFull, fk, (__ffs(bins) - 1) & 31) != (int32_t)f) continue;  // another bin's item does it
        int32_t lo = INT32_MAX, hi = 0;  // the widest window
        int32_t blo[NB ? NB : 1];
        uint32_t wid[NB ? NB : 1];
        if constexpr (NB > 0) {
#pragma unroll
            for (int k = 0; k < NB; ++k) {
                const bool on = (bins >> k) & 1u;
                blo[k] = on ? s_lo[k] + 1 : 0;
                wid[k] = on ? (uint32_t)(s_hi[k] - s_lo[k]) : 0u;
                if (on) lo = min(lo, s_lo[k]), hi = max(hi, s_hi[k]);
            }
        } else {
            for (unsigned b = bins; b; b &= b - 1) {
                lo = min(lo, s_lo[__ffs(b) - 1]);
                hi = max(hi, s_hi[__ffs(b) - 1]);
            }
        }
        auto bins_of = [&](int32_t d) {  // the bins that distance d lies in
            unsigned m = 0;
            if constexpr (NB > 0) {
#pragma unroll
                for (int k = 0; k < NB; ++k)
                    if ((uint32_t)(d - blo[k]) < wid[k]) m |= 1u << k;
            } else {
                for (unsigned b = bins; b; b &= b - 1) {
                    const int k = __ffs(b) - 1;
                    if (s_lo[k] < d && d <= s_hi[k]) m |= 1u << k;
                }
            }
            return m;
        };
        // where lane k's bin keeps its bitsets
        const int64_t wb = a.base[r] + ((int64_t)fk - a.f2foff[r]) * (int64_t)a.stride[r];
        auto put = [&](uint32_t *bits, int b, unsigned m) {  // lane k writes bin k's word
            uint32_t w = 0;
            if constexpr (NB > 0) {
#pragma unroll
                for (int k = 0; k < NB; ++k) {
                    const unsigned v = __ballot_sync(kFull, (m >> k) & 1u);
                    if (lane == k) w = v;
                }
            } else {
                for (unsigned q = bins; q; q &= q - 1) {
                    const int k = __ffs(q) - 1;
                    const unsigned v = __ballot_sync(kFull, (m >> k) & 1u);
                    if (lane == k) w = v;
                }
            }
            if (fk >= 0) bits[wb + (b >> 5)] = w;
        };
        const int32_t *tlX = ri.ttime + xb;
        const int32_t *tlY = ri.ttime + yb;
        // V: a Y event at t is a valid end of bin (lo, hi] when an X event lies
        // in [t - hi, t - lo)
        {
            const int32_t *row = ri.tidx + (int64_t)X * (ri.tcells + 1);
            for (int b = b0; b < lenY && b < b1; b += 32) {
                unsigned m = 0;
                const int32_t t = b + lane < lenY ? tlY[b + lane] : 0;
                if (t > lo) {
                    const int32_t from = max(t - hi, 0), to = t - lo;
                    for (int pos = cell_of(ri, row, (uint32_t)from); pos < lenX; ++pos) {
                        const int32_t x = tlX[pos];
                        if (x >= to) break;
                        if (x >= from) m |= bins_of(t - x);
                    }
                }
                put(a.vbits, b, m);
            }
        }
        // S: an X event at t is a valid start when a Y event lies in
        // (t + lo, t + hi]
        {
            const int32_t *row = ri.tidx + (int64_t)Y * (ri.tcells + 1);
            for (int b = b0; b < lenX && b < b1; b += 32) {
                unsigned m = 0;
                if (b + lane < lenX) {
                    const uint32_t t = (uint32_t)tlX[b + lane], from = t + (uint32_t)lo + 1u, to = t + (uint32_t)hi;
                    for (int pos = cell_of(ri, row, from); pos < lenY; ++pos) {
                        const uint32_t x = (uint32_t)tlY[pos];
                        if (x > to) break;
                        if (x >= from) m |= bins_of((int32_t)(x - t));
                    }
                }
                put(a.sbits, b, m);
            }
        }
    }
}

// One warp per level-3 candidate: UB, and the skip flag when UB is at or
// below the threshold (or-ed into the flags another bound set, if any);
// skipped candidates are counted per recording.
__global__ void k_jb_bound(JoinBoundArgs a) {
    const int lane = threadIdx.x & 31;
    const int64_t C = *a.cn;
    const bool usable = a.base[a.n_recs] <= a.cap_words;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t c = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; c < C; c += nw) {
        const uint32_t r = a.crec[c];
        bool sk = false;
        if (usable) {
            const uint32_t A = a.ct[3 * c], B = a.ct[3 * c + 1], Cc = a.ct[3 * c + 2];
            const int k1 = bin_of(a, a.cl[2 * c], a.ch[2 * c]), k2 = bin_of(a, a.cl[2 * c + 1], a.ch[2 * c + 1]);
            const int64_t to = a.tab_off[r];
            const int64_t nt = a.nt[r];
            const int32_t f1 = k1 < a.nb ? a.tab[to + ((int64_t)A * nt + B) * a.nb + k1] : -1;
            const int32_t f2 = k2 < a.nb ? a.tab[to + ((int64_t)B * nt + Cc) * a.nb + k2] : -1;
            if (f1 >= 0 && f2 >= 0) {
                const RecInfo &ri = a.ri[r];
                const int lenB = (int)(ri.toff[B + 1] - ri.toff[B]);
                const int64_t st = a.stride[r];
                const uint32_t *v = a.vbits + a.base[r] + (f1 - a.f2foff[r]) * st;
                const uint32_t *s = a.sbits + a.base[r] + (f2 - a.f2foff[r]) * st;
                uint32_t acc = 0;
                for (int w = lane; w < (lenB + 31) >> 5; w += 32) acc += __popc(v[w] & s[w]);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
                sk = acc <= a.thr[r];
            }
        }
        if (lane == 0) {
            const bool fin = sk || (a.or_skip && a.skip[c]);
            a.skip[c] = fin ? 1 : 0;
            if (fin) atomicAdd(a.skipc + r, 1ull);
        }
    }
}

}  // namespace

int join_bound_level3(cudaStream_t st, int n_sm, const JoinBoundArgs &a) {
    const unsigned g = (unsigned)std::max(1, 8 * n_sm);
    if (cudaMemsetAsync(a.tab, 0xFF, sizeof(int32_t) * (size_t)std::max<int64_t>(a.tab_n, 1), st) != cudaSuccess ||
        cudaMemsetAsync(a.skipc, 0, sizeof(unsigned long long) * (size_t)std::max(a.n_recs, 1), st) != cudaSuccess)
        return FEM_ERR_CUDA;
    k_jb_index<<<g, 256, 0, st>>>(a);
    k_jb_base<<<1, 32, 0, st>>>(a);
    // one wave of resident blocks: a second would start with the largest
    // recordings' items left over
    if (a.nb <= 4)
        k_jb_bits<4><<<6 * std::max(1, n_sm), 256, 0, st>>>(a);
    else
        k_jb_bits<0><<<6 * std::max(1, n_sm), 256, 0, st>>>(a);
    k_jb_bound<<<g, 256, 0, st>>>(a);
    FEM_CUDA_TRY(cudaGetLastError());
    return FEM_OK;
}

}  // namespace fem
