// Parts of a selection that the cluster launches share (refine_loop.cu, tail.cu): the threshold search over
// the gain histogram, the sort of the rebalance's candidates and the prefix they move.
//
// The launches loop over short phases that a few thousand cycles of work separate, so their code is kept small:
// loops that do not need it are not unrolled and these functions are not inlined.  With them inlined and
// unrolled by the compiler the loop was 150 KB of code and every phase began with 1,000 to 2,000 cycles of
// instruction fetch.
#pragma once

#include <climits>

#include "common.cuh"
#include "refine_dev.cuh"

namespace bp {

struct FindScratch {
    unsigned wsum[2][16], bin[2], above[2];
    unsigned slow;  // a group needs the exact radix passes
    unsigned hit;   // the threshold is the guessed gain
};

// Block-wide sum and exclusive prefix of 32-bit values (node counts, node weights: every total of a hypergraph
// stays below 2^31).  red: one entry per warp.
template <int kT>
__device__ __noinline__ unsigned block_sum32(unsigned v, unsigned *red) {
    static_assert(kT <= 1024, "one lane per warp sum");
    const int lane = threadIdx.x & 31;
    v = __reduce_add_sync(0xffffffffu, v);
    __syncthreads();
    if (lane == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    return __reduce_add_sync(0xffffffffu, lane < kT / 32 ? red[lane] : 0u);
}
template <int kT>
__device__ __noinline__ unsigned block_scan32(unsigned v, unsigned *red, unsigned *total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned inc = warp_inclusive_scan(v);
    __syncthreads();
    if (lane == 31) red[wid] = inc;
    __syncthreads();
    const unsigned s = lane < kT / 32 ? red[lane] : 0u;
    *total = __reduce_add_sync(0xffffffffu, s);
    return __reduce_add_sync(0xffffffffu, lane < wid ? s : 0u) + inc - v;
}

// d_sel_find's decision from the histogram's totals with three barriers.  Half of the block searches each
// group: a thread sums eight bins, every warp adds up the warps above it, the warp holding the threshold
// searches its bins.  With a guess, `ties` candidates sit at the guessed `gain` and the histogram holds those
// above it; returns false when the threshold lies below the guess.
template <int kT>
__device__ __noinline__ bool find_threshold(RState *st, FindScratch &s, int kind, long long sq, bool guess, int gain,
                                            unsigned ties) {
    constexpr int kHalf = kT / 2, kPer = kHistBins / kHalf, kW = kHalf / 32;
    static_assert(kPer == 8, "two uint4 of bins per thread");
    const int lane = threadIdx.x & 31;
    const int i = (int)threadIdx.x >= kHalf, t = (int)threadIdx.x - i * kHalf, w = t >> 5;
    const int b0 = kHistBins - kPer * (t + 1);  // this thread's bins, taken from the highest down
    const unsigned *hist = &st->hist[i][b0];
    const uint4 lo = *reinterpret_cast<const uint4 *>(hist), hi = *reinterpret_cast<const uint4 *>(hist + 4);
    const unsigned own = lo.x + lo.y + lo.z + lo.w + hi.x + hi.y + hi.z + hi.w;
    const unsigned sum = __reduce_add_sync(0xffffffffu, own);
    if (lane == 0) s.wsum[i][w] = sum;
    if (t == 0) s.bin[i] = ~0u;
    if (threadIdx.x == 0) s.slow = 0;
    __syncthreads();
    const unsigned c = lane < kW ? s.wsum[i][lane] : 0u;
    const unsigned cnt = __reduce_add_sync(0xffffffffu, c);
    const unsigned other = __reduce_add_sync(0xffffffffu, lane < kW ? s.wsum[i ^ 1][lane] : 0u);
    const unsigned before = __reduce_add_sync(0xffffffffu, lane < w ? c : 0u);
    const int heavy = st->heavy, grp = kind == SEL_INITIAL ? 1 : heavy;
    bool hit = false;
    unsigned K = 0;
    if (kind == SEL_REFINE) {
        K = min(cnt, other);
    } else {
        const long long have = grp == i ? cnt : other;  // of the group selected from
        if (guess && have < sq) {
            if (have + ties < sq) return false;  // the same in every thread and block
            hit = true;
        }
        if (grp == i) K = (unsigned)min(have, sq);
    }
    const unsigned need = !hit && K > 0 && K < cnt ? K : 0u;
    if (need > before && need <= before + sum) {  // this warp's bins hold the need-th key
        unsigned run = before + warp_inclusive_scan(own) - own;
        if (need > run && need <= run + own) {
            int k = kPer - 1;
#pragma unroll 1
            for (; k > 0 && need > run + hist[k]; --k) run += hist[k];
            s.bin[i] = (unsigned)(b0 + k);
            s.above[i] = run;
        }
    }
    __syncthreads();
    if (t == 0) {
        SelGroup &G = st->g[i];
        G.cnt = cnt;
        G.K = K;
        const int b = (int)s.bin[i];
        if (hit && i == heavy) {
            G.mode = 2;
            G.thr = gkey(gain);
            G.take_eq = (unsigned)(sq - (long long)cnt);
        } else if (K == 0) {
            G.mode = 0;
        } else if (K >= cnt) {
            G.mode = 1;
        } else if (b > 0 && b < kHistBins - 1) {
            G.mode = 2;
            G.thr = gkey(b + kClampLo);
            G.take_eq = K - s.above[i];
        } else {
            // the threshold lies in a clamped end bucket: exact radix select over its keys
            const bool top = b == kHistBins - 1;
            G.mode = 3;
            G.need = K - s.above[i];
            G.base = top ? gkey(kHistBins - 1 + kClampLo) : 0u;
            G.top = top ? 1ull << 32 : (unsigned long long)gkey(kClampLo) + 1ull;
            const unsigned long long range = G.top - G.base;
            const unsigned bits = range > 1 ? 64 - __clzll(range - 1ull) : 0;
            G.shift = bits > kHistBits ? bits - kHistBits : 0;
            s.slow = 1;
        }
        if (i == 0) s.hit = hit;
    }
    __syncthreads();
    return true;
}

// Sorts keys[0, S) ascending (S a power of two): in registers with warp shuffles where a thread holds
// one key, in shared memory above.
template <int kT>
__device__ __noinline__ void sort_keys(unsigned long long *keys, int S) {
    const int t = threadIdx.x;
    if (S <= kT) {
        unsigned long long k0 = t < S ? keys[t] : ~0ull;
#pragma unroll 1
        for (int k = 2; k <= S; k <<= 1) {
            const bool up = (t & k) == 0;
#pragma unroll 1
            for (int j = k >> 1; j > 0; j >>= 1) {
                unsigned long long o;
                if (j >= 32) {
                    __syncthreads();
                    if (t < S) keys[t] = k0;
                    __syncthreads();
                    o = t < S ? keys[t ^ j] : ~0ull;
                } else {
                    o = __shfl_xor_sync(0xffffffffu, k0, j);
                }
                const bool lower = (t & j) == 0;
                k0 = (lower == up) == (o < k0) ? o : k0;
            }
        }
        __syncthreads();
        if (t < S) keys[t] = k0;
        __syncthreads();
        return;
    }
#pragma unroll 1
    for (int k = 2; k <= S; k <<= 1)
#pragma unroll 1
        for (int j = k >> 1; j > 0; j >>= 1) {
#pragma unroll 1
            for (int i = t; i < S; i += kT) {
                const int q = i ^ j;
                if (q > i) {
                    const unsigned long long u = keys[i], v = keys[q];
                    if ((u > v) == ((i & k) == 0)) { keys[i] = v; keys[q] = u; }
                }
            }
            __syncthreads();
        }
}

struct CutScratch {
    int cut;
    unsigned moved;
};

// The rebalance's prefix (reading C13) of keys[0, n), keys = gain descending << 32 | node, total weight `total`:
// the shortest by (gain descending, id ascending) that reaches `need`, of at most sq nodes, stopping before the
// node that would exceed `room`.  All threads; returns its length, its weight in *moved.  When all candidates
// together do not reach `need` (most rounds) they all move and the keys stay unsorted.
template <int kT>
__device__ __noinline__ int rebal_prefix(unsigned long long *keys, int n, long long sq, long long room, long long need,
                                         const int *nw, unsigned total, unsigned *red, CutScratch &s, unsigned *moved) {
    int cut = (int)min((long long)n, sq);
    *moved = total;
    if (total < need && total <= room && cut == n) return cut;
    int S = 1;
    while (S < n) S <<= 1;
    if (threadIdx.x == 0) {
        s.cut = cut;
        s.moved = total;
    }
    sort_keys<kT>(keys, S);
    // every thread a run of consecutive nodes; the first node past room, or the first to reach need,
    // ends the prefix, and its thread knows the weight before or up to it
    const int per = (n + kT - 1) / kT, i0 = min((int)threadIdx.x * per, n), i1 = min(i0 + per, n);
    unsigned loc = 0, tot;
#pragma unroll 1
    for (int i = i0; i < i1; ++i) loc += (unsigned)nw[(unsigned)keys[i]];
    unsigned run = block_scan32<kT>(loc, red, &tot), at = 0;
    int mine = -1;
#pragma unroll 1
    for (int i = i0; i < i1; ++i) {
        const unsigned up = run + (unsigned)nw[(unsigned)keys[i]];
        if (up > room || up >= need) {
            const bool over = up > room;  // node i would exceed room: it stays
            mine = i + !over;
            at = over ? run : up;
            atomicMin(&s.cut, mine);
            break;
        }
        run = up;
    }
    __syncthreads();
    cut = s.cut;
    if (mine == cut) s.moved = at;
    __syncthreads();
    *moved = s.moved;
    return cut;
}

}  // namespace bp
