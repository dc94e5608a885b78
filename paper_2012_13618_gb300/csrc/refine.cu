// Initial partitioning and refinement on sm_103a (Sec. 3.2-3.3): Algorithm 4 move gains from
// per-hyperedge side counts, Algorithm 3 growth of P0 by the top ceil(sqrt n) gains, Algorithm 5
// swaps of the gain >= 0 lists and the rebalancing pass.
//
// Per level: k_level_start (sides projected, accumulators reset), k_hedge_n1 (pins per side of every
// hyperedge), k_node_gain (gains), all over the whole grid, then one cluster launch that runs the
// level's selections, moves and loops (refine_loop.cu) and keeps the gains current from the moved
// nodes.  A selection that moves too many incidences for one cluster stops that launch; the grid
// brings the gains up to date (k_move_pairs, k_move_gains) and the cluster launch goes on.  A
// captured bisection replays the recorded stops as straight-line kernels and verifies them.
//
// Node order is always (gain descending, node id ascending).  A top-K is found without sorting:
// one histogram pass over gains clamped to [-1024, 1023] fixes the threshold gain exactly unless
// it falls in one of the two clamped end buckets, in which case an exact radix select (up to
// three 11-bit passes over the order-preserving key gain ^ 0x80000000) narrows it down; the lowest
// ids among nodes whose gain equals the threshold are then taken.  Only the rebalancing pass needs the
// chosen nodes in order; it sorts at most ceil(sqrt n) of them.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstddef>

#include "common.cuh"
#include "internal.h"
#include "lb.cuh"
#include "move_dev.cuh"
#include "refine_dev.cuh"
#include "refine_loop.h"
#include "select_dev.cuh"

namespace bp {

namespace {

constexpr int kBlock = 256;

inline int grid_for(int64_t n, int per_block = kBlock, int cap = 152 * 16) {
    int64_t b = (n + per_block - 1) / per_block;
    if (b < 1) b = 1;
    return (int)std::min<int64_t>(b, cap);
}

// Levels whose nodes average more incidences than this sum each warp's gain flushes per node
// before the atomic (many threads end on one node there); on the others it only costs time.
constexpr int kWarpSumDegree = 64;

}  // namespace

// Start of a level's refinement: the coarser level's sides projected (the coarsest level: all nodes
// on side 1), the gains and the loop state zero, every hyperedge's pins counted on side 0.
__global__ void __launch_bounds__(kBlock)
k_level_start(int N, int E, const int *__restrict__ cmap, const uint8_t *__restrict__ coarse,
              uint8_t *__restrict__ side, uint8_t *__restrict__ prev, int *__restrict__ gain,
              const int *__restrict__ hoff, unsigned long long *__restrict__ pair, LoopState *ls) {
    const int n = E > N ? E : N;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        if (i < N) {
            const uint8_t s = cmap ? __ldg(coarse + __ldg(cmap + i)) : (uint8_t)1;
            side[i] = s;
            prev[i] = s;
            gain[i] = 0;
        }
        if (i < E) pair[i] = (unsigned long long)(unsigned)(__ldg(hoff + i + 1) - __ldg(hoff + i)) << 32;
    }
    if (blockIdx.x == 0)
        for (int i = threadIdx.x; i < (int)(offsetof(LoopState, cmd) / sizeof(unsigned)); i += blockDim.x)
            reinterpret_cast<unsigned *>(ls)[i] = 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) ls->sel = ls->it = ls->rebal = ls->go = ls->ticket = 0;
}

__global__ void __launch_bounds__(kLbBlock)
k_hedge_n1(int E, int P, const int *__restrict__ hoff, const int *__restrict__ pins,
           const uint8_t *__restrict__ side, unsigned long long *__restrict__ pair,
           const int *__restrict__ ts) {
    d_hedge_n1(GridTeam(), E, P, hoff, pins, side, pair, ts);
}

__global__ void __launch_bounds__(kLbBlock)
k_node_gain(int N, int P, const int *__restrict__ noff, const int *__restrict__ nadj,
            const unsigned long long *__restrict__ pair, const int *__restrict__ hw,
            const uint8_t *__restrict__ side, int *__restrict__ gain, const int *__restrict__ ts,
            bool warp_sum) {
    d_node_gain(GridTeam(), N, P, noff, nadj, pair, hw, side, gain, ts, warp_sum);
}

// The grid's part of a large move (move_dev.cuh): pass 1, then pass 2.  Above P / kMoveFull (kMoveFullHubs)
// moved incidences only the pairs are updated and every gain is recomputed from them.
__device__ __forceinline__ bool move_full(const MoveArgs &m, const LoopRound *rd) {
    const int part = (long long)m.P >= (long long)kHubDegree * m.N ? kMoveFullHubs : kMoveFull;
    return (long long)__ldcg(&rd->inc) * part > (long long)m.P;
}

// grid_sel: after a selection by the grid, which may not have taken place.
__global__ void __launch_bounds__(kBlock) k_move_pairs(MoveArgs m, bool grid_sel) {
    if (grid_sel && !__ldcg(&m.ls->go)) return;
    LoopRound *rd = &m.ls->rd[m.ls->sel];
    const int tid = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
    const bool full = move_full(m, rd);
    if (blockIdx.x == 0) {  // clear for the next selection (neither pass reads them)
        unsigned *h = &m.ls->hist[0][0], *other = reinterpret_cast<unsigned *>(&m.ls->rd[m.ls->sel ^ 1]);
        for (int i = threadIdx.x; i < 2 * kHistBins; i += blockDim.x) h[i] = 0;
        for (int i = threadIdx.x; i < (int)(sizeof(LoopRound) / sizeof(unsigned)); i += blockDim.x) other[i] = 0;
    }
    if (full)
        for (int v = tid; v < m.N; v += nt) m.gain[v] = 0;
    move_pass1(m, __ldcg(&rd->ents), &rd->items, tid >> 5, nt >> 5, m.prev, full);
}

__global__ void __launch_bounds__(kLbBlock) k_move_gains(MoveArgs m, const int *__restrict__ ts, bool warp_sum,
                                                         bool grid_sel) {
    if (grid_sel && !__ldcg(&m.ls->go)) return;
    const LoopRound *rd = &m.ls->rd[m.ls->sel];
    if (move_full(m, rd)) {
        d_node_gain(GridTeam(), m.N, m.P, m.noff, m.nadj, m.pair, m.hw, m.side, m.gain, ts, warp_sum);
        return;
    }
    const int tid = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
    move_pass2(m, __ldcg(&rd->ents), __ldcg(&rd->items), tid >> 5, nt >> 5, m.prev, true);
}

// A refinement selection (Algorithm 5) by the whole grid in three launches: k_sel_count (the gains' histogram; the
// last block finds the thresholds), k_sel_apply (nodes above them flipped and listed, ties counted per block), k_sel_ties
// (the ties of lowest ids).  One cluster streams a level's nodes at a few hundred GB/s and lists a few nodes a
// cycle; where many nodes move that was most of an iteration (5M-node row-net: 1 ms a selection, 0.2 so).  Nothing is read back: a
// threshold in a clamped end bucket leaves this and the following selections of the level to the cluster launch
// (`go`), which goes on with iteration ls->it in any case.
constexpr int kSelBlock = 512, kSelBlocks = 304, kSelStep = 8 * kSelBlock;

// The block's nodes [lo, hi).
__device__ __forceinline__ void sel_range(int N, int &lo, int &hi) {
    const int R = (int)(((long long)N + gridDim.x - 1) / gridDim.x + 31) & ~31;
    lo = (int)min((long long)R * blockIdx.x, (long long)N);
    hi = (int)min((long long)lo + R, (long long)N);
}

// Gains of the thread's eight consecutive nodes from v (a multiple of 8), the lowest value from `hi` on, and
// their sides as bits (0 where no gain is at least `floor`).
__device__ __forceinline__ unsigned sel_load(const MoveArgs &m, const uint8_t *sides, int v, int hi, int floor, int *g) {
#pragma unroll
    for (int q = 0; q < 8; ++q) g[q] = INT_MIN;
    if ((unsigned)v >= (unsigned)hi) return 0;
    const int4 a = __ldcg(reinterpret_cast<const int4 *>(m.gain + v));
    g[0] = a.x;
    if (v + 1 < hi) g[1] = a.y;
    if (v + 2 < hi) g[2] = a.z;
    if (v + 3 < hi) g[3] = a.w;
    if (v + 4 < hi) {
        const int4 b = __ldcg(reinterpret_cast<const int4 *>(m.gain + v + 4));
        g[4] = b.x;
        if (v + 5 < hi) g[5] = b.y;
        if (v + 6 < hi) g[6] = b.z;
        if (v + 7 < hi) g[7] = b.w;
    }
    int top = g[0];
#pragma unroll
    for (int q = 1; q < 8; ++q) top = max(top, g[q]);
    if (top < floor) return 0;
    unsigned on1 = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q)
        if (v + q < hi && __ldcg(sides + v + q)) on1 |= 1u << q;
    return on1;
}

// The nodes v + q of the mask flip and join the move list (all threads of the block); on1: their sides so far.
__device__ __forceinline__ void sel_take(const MoveArgs &m, LoopRound *rd, int v, unsigned mask, unsigned on1,
                                         unsigned *red, unsigned *base, unsigned &inc, int &weight) {
    int b[8], d[8];
    unsigned own = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const bool in = mask >> q & 1u;
        b[q] = in ? __ldg(m.noff + v + q) : 0;
        d[q] = in ? __ldg(m.noff + v + q + 1) : 0;
        const int w = in ? __ldg(m.nw + v + q) : 0;
        weight += on1 >> q & 1u ? -w : w;
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        d[q] -= b[q];
        inc += (unsigned)d[q];
        if (mask >> q & 1u) {
            m.side[v + q] = (uint8_t)(on1 >> q & 1u ^ 1u);
            own += d[q] > 0 ? ((unsigned)d[q] + (unsigned)m.run - 1u) >> m.run_shift : 1u;
        }
    }
    unsigned tot;
    const unsigned ex = block_scan32<kSelBlock>(own, red, &tot);
    if (threadIdx.x == 0) *base = tot ? atomicAdd(&rd->ents, tot) : 0u;
    __syncthreads();
    unsigned o = *base + ex;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const bool in = mask >> q & 1u;
        const int side = (int)(on1 >> q & 1u ^ 1u);
        const unsigned c = !in ? 0u : (d[q] > 0 ? ((unsigned)d[q] + (unsigned)m.run - 1u) >> m.run_shift : 1u);
        if (c <= 8)
#pragma unroll 1
            for (unsigned i = 0; i < c; ++i) m.ent[o + i] = move_entry(v + q, b[q], d[q], (int)i, side, m.run);
        unsigned hubs = __ballot_sync(0xffffffffu, c > 8);  // long lists: the warp together
        while (hubs) {
            const int src = __ffs(hubs) - 1;
            hubs &= hubs - 1;
            const int hv = __shfl_sync(0xffffffffu, v + q, src), hb = __shfl_sync(0xffffffffu, b[q], src);
            const int hd = __shfl_sync(0xffffffffu, d[q], src), hs = __shfl_sync(0xffffffffu, side, src);
            const unsigned ho = __shfl_sync(0xffffffffu, o, src), hc = __shfl_sync(0xffffffffu, c, src);
#pragma unroll 1
            for (unsigned i = threadIdx.x & 31; i < hc; i += 32) m.ent[ho + i] = move_entry(hv, hb, hd, (int)i, hs, m.run);
        }
        o += c;
    }
    __syncthreads();
}

// The block's sums join the round's and the side weights.
__device__ __forceinline__ void sel_sums(LoopState *ls, LoopRound *rd, unsigned inc, int weight) {
    inc = __reduce_add_sync(0xffffffffu, inc);
    weight = __reduce_add_sync(0xffffffffu, weight);
    if ((threadIdx.x & 31) != 0) return;
    if (inc) atomicAdd(&rd->inc, (unsigned long long)inc);
    if (weight) {
        atomicAdd(&ls->W[1], (unsigned long long)(long long)weight);
        atomicAdd(&ls->W[0], (unsigned long long)-(long long)weight);
    }
}

__global__ void __launch_bounds__(kSelBlock) k_sel_count(MoveArgs m, int it) {
    __shared__ __align__(16) RState st;
    __shared__ FindScratch find;
    __shared__ bool last;
    LoopState *ls = m.ls;
    if ((int)__ldcg(&ls->it) != it) {  // an earlier selection was left to the cluster
        if (blockIdx.x == 0 && threadIdx.x == 0) ls->go = 0;
        return;
    }
    // the last selection's moves are in the gains: the sides before this one
    move_settle(m, __ldcg(&ls->rd[__ldcg(&ls->sel)].ents), blockIdx.x * kSelBlock + threadIdx.x, gridDim.x * kSelBlock);
    unsigned *h = &st.hist[0][0];
    for (int i = threadIdx.x; i < 2 * kHistBins; i += kSelBlock) h[i] = 0;
    __syncthreads();
    int lo, hi;
    sel_range(m.N, lo, hi);
    for (int v0 = lo; v0 < hi; v0 += kSelStep) {
        int g[8];
        const unsigned on1 = sel_load(m, m.side, v0 + 8 * (int)threadIdx.x, hi, 0, g);
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (g[q] >= 0) atomicAdd(&st.hist[on1 >> q & 1u][min(g[q], kHistBins - 1 + kClampLo) - kClampLo], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * kHistBins; i += kSelBlock)
        if (h[i]) atomicAdd(&ls->hist[0][0] + i, h[i]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&ls->ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int i = threadIdx.x; i < 2 * kHistBins; i += kSelBlock) h[i] = __ldcg(&ls->hist[0][0] + i);
    if (threadIdx.x == 0) st.heavy = -1;
    __syncthreads();
    find_threshold<kSelBlock>(&st, find, SEL_REFINE, 0, false, 0, 0);
    const bool slow = find.slow != 0;
    if (threadIdx.x == 0) {
        ls->ticket = 0;
        ls->go = !slow;
        if (!slow) ls->sel ^= 1u;
    }
    if (threadIdx.x < 2) {
        const SelGroup &G = st.g[threadIdx.x];
        ls->mode[threadIdx.x] = G.mode;
        ls->thr[threadIdx.x] = G.thr;
        ls->take[threadIdx.x] =
            G.mode == 2 && !slow && st.hist[threadIdx.x][(int)(G.thr ^ 0x80000000u) - kClampLo] > G.take_eq ? G.take_eq : 0u;
    }
    if (slow)
        for (int i = threadIdx.x; i < 2 * kHistBins; i += kSelBlock) (&ls->hist[0][0])[i] = 0;
}

__global__ void __launch_bounds__(kSelBlock) k_sel_apply(MoveArgs m, unsigned *__restrict__ ties) {
    __shared__ unsigned red[32], base, n_tie[2];
    LoopState *ls = m.ls;
    if (!__ldcg(&ls->go)) return;
    LoopRound *rd = &ls->rd[__ldcg(&ls->sel)];
    const unsigned mode0 = __ldcg(&ls->mode[0]), mode1 = __ldcg(&ls->mode[1]);
    const unsigned thr0 = __ldcg(&ls->thr[0]), thr1 = __ldcg(&ls->thr[1]);
    const bool some0 = __ldcg(&ls->take[0]) != 0, some1 = __ldcg(&ls->take[1]) != 0;
    if (threadIdx.x < 2) n_tie[threadIdx.x] = 0;
    __syncthreads();
    int lo, hi, weight = 0;
    unsigned inc = 0, t0 = 0, t1 = 0;
    sel_range(m.N, lo, hi);
    for (int v0 = lo; v0 < hi; v0 += kSelStep) {
        int g[8];
        const int v = v0 + 8 * (int)threadIdx.x;
        const unsigned on1 = sel_load(m, m.side, v, hi, 0, g);
        unsigned mask = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            if (g[q] < 0) continue;
            const bool one = on1 >> q & 1u;
            const unsigned k = gkey(g[q]), mode = one ? mode1 : mode0, thr = one ? thr1 : thr0;
            const bool tie = mode == 2 && k == thr && (one ? some1 : some0);
            if (tie) ++(one ? t1 : t0);
            else if (mode == 1 || (mode == 2 && k >= thr)) mask |= 1u << q;
        }
        sel_take(m, rd, v, mask, on1, red, &base, inc, weight);
    }
    sel_sums(ls, rd, inc, weight);
    t0 = __reduce_add_sync(0xffffffffu, t0);
    t1 = __reduce_add_sync(0xffffffffu, t1);
    if ((threadIdx.x & 31) == 0 && (t0 | t1)) {
        atomicAdd(&n_tie[0], t0);
        atomicAdd(&n_tie[1], t1);
    }
    __syncthreads();
    if (threadIdx.x < 2) ties[2 * blockIdx.x + threadIdx.x] = n_tie[threadIdx.x];
}

__global__ void __launch_bounds__(kSelBlock) k_sel_ties(MoveArgs m, const unsigned *__restrict__ ties, int it) {
    static_assert(kSelBlocks <= kSelBlock, "one thread per block's ties");
    __shared__ unsigned red[32], base;
    LoopState *ls = m.ls;
    if (!__ldcg(&ls->go)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) ls->it = (unsigned)it + 1u;
    LoopRound *rd = &ls->rd[__ldcg(&ls->sel)];
    int lo, hi, weight = 0;
    unsigned inc = 0;
    sel_range(m.N, lo, hi);
    for (int i = 0; i < 2; ++i) {
        const unsigned want = __ldcg(&ls->take[i]);
        if (want == 0) continue;  // the same in every block
        const unsigned before = block_sum32<kSelBlock>((int)threadIdx.x < (int)blockIdx.x ? ties[2 * threadIdx.x + i] : 0u, red);
        const unsigned own = ties[2 * blockIdx.x + i];
        const unsigned take = before >= want ? 0u : min(own, want - before);
        const int thr = (int)(__ldcg(&ls->thr[i]) ^ 0x80000000u);
        unsigned run = 0;
        for (int v0 = lo; v0 < hi && run < take; v0 += kSelStep) {
            int g[8];
            const int v = v0 + 8 * (int)threadIdx.x;
            const unsigned on1 = sel_load(m, m.prev, v, hi, thr, g);  // the sides before this selection
            unsigned tie = 0, tot;
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (g[q] == thr && (int)(on1 >> q & 1u) == i) tie |= 1u << q;
            unsigned rank = run + block_scan32<kSelBlock>((unsigned)__popc(tie), red, &tot), mask = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (tie >> q & 1u) {
                    if (rank < take) mask |= 1u << q;
                    ++rank;
                }
            __syncthreads();
            sel_take(m, rd, v, mask, i ? 255u : 0u, red, &base, inc, weight);
            run += tot;
        }
        __syncthreads();
    }
    sel_sums(ls, rd, inc, weight);
}

// ------------------------------------------------------------------------ host side
int64_t balance_limit(int64_t W, int32_t ms, int32_t m, int64_t e6) {
    const __int128 share = (__int128)W * ms;  // the side's share is share / m
    const int64_t a = (int64_t)((share + m - 1) / m);
    const int64_t b = (int64_t)(share * (1000000 + e6) / ((__int128)m * 1000000));
    return a > b ? a : b;
}

static int64_t ceil_sqrt64(int64_t n) {
    if (n <= 0) return 0;
    int64_t r = (int64_t)sqrt((double)n);
    while (r * r > n) r--;
    while ((r + 1) * (r + 1) <= n) r++;
    return r * r == n ? r : r + 1;
}

namespace {

// The refinement state in the handle's small scratch.
LoopState *loop_state(bipart_graph *g) {
    return reinterpret_cast<LoopState *>(g->w.small.as<char>() + 256);
}

// Nodes with short incidence lists share a warp four at a time.
bool short_lists(const Level &L) { return (int64_t)L.P <= kMoveRunShort * (int64_t)L.N; }

// A level's refinement from the sides in `side` (k_level_start projects them from `coarse`, the
// sides of the next coarser level; null: the coarsest level, with Algorithm 3 first).
void refine_level(bipart_graph *g, Level &L, const int *cmap, const uint8_t *coarse, int coarse_n, uint8_t *side,
                  LoopParams p) {
    cudaStream_t s = g->stream;
    Work &w = g->w;
    LoopState *ls = loop_state(g);
    MoveArgs m{};
    m.N = L.N; m.E = L.E; m.P = L.P;
    m.noff = L.noff(); m.nadj = L.nadj(); m.hoff = L.hoff(); m.pins = L.pins(); m.hw = L.hw(); m.nw = L.nw();
    m.side = side;
    m.prev = w.side_prev.as<uint8_t>();
    m.gain = w.n_c.as<int>();
    m.pair = w.pair.as<unsigned long long>();
    m.ls = ls;
    m.ent = w.n_key.as<int4>();
    m.items = w.items.as<int4>();
    m.item_cap = kItemCap;
    const bool shorter = short_lists(L);
    m.lanes = shorter ? 8 : 32;
    m.run = shorter ? kMoveRunShort : kMoveRun;
    m.run_shift = shorter ? 4 : 6;
    p.sq = ceil_sqrt64(L.N);
    if (p.sq > kRebalMax) throw Fail{BIPART_ERR_OOM, "level too large for the ordered rebalance"};
    auto *cand = (unsigned long long *)w.list.ensure(sizeof(unsigned long long) * (size_t)std::max<int64_t>(p.sq, 1), s);
    const bool warp_sum = (int64_t)L.P > kWarpSumDegree * (int64_t)L.N;
    p.start = L.P <= kLoopStartPins && L.N <= kLoopStartNodes;
    p.cmap = cmap;
    p.coarse = coarse;
    if (!p.start) {
        {
            ProfScope ps("project", 11.0 * L.N + 12.0 * L.E, s);
            k_level_start<<<grid_for(std::max(L.N, L.E)), kBlock, 0, s>>>(L.N, L.E, cmap, coarse, side, m.prev,
                                                                          m.gain, m.hoff, m.pair, ls);
            BP_LAUNCH();
        }
        if (L.P > 0) {
            // hoff, pins, one side byte per pin, one atomic per hyperedge run
            ProfScope ps("hedge_n1", 8.0 * L.E + 5.0 * L.P, s);
            k_hedge_n1<<<lb_grid(L.P), kLbBlock, 0, s>>>(L.E, L.P, L.hoff(), L.pins(), side, m.pair, L.tsh());
            BP_LAUNCH();
        }
        if (L.P > 0) {
            // noff, nadj, 8-byte pair gather per incidence (and a weight where it counts), side, gain
            ProfScope ps("node_gain", 9.0 * L.N + 12.0 * L.P, s);
            k_node_gain<<<lb_grid(L.P), kLbBlock, 0, s>>>(L.N, L.P, L.noff(), L.nadj(), m.pair, L.hw(), side, m.gain,
                                                           L.tsn(), warp_sum);
            BP_LAUNCH();
        }
    }
    p.suspend = L.P > kLoopAlonePins || L.N > kGridSelLarge;
    p.resume = false;
    if (p.suspend && !p.initial && (L.N > kGridSelLarge || (L.N > kGridSelNodes && L.N / kGridSelRatio >= coarse_n))) {
        auto *ties = reinterpret_cast<unsigned *>(cand);  // the rebalance's candidates come later
        static_assert((long long)kSelBlocks * kSelBlocks <= kGridSelNodes, "2 ties a block fit the sqrt(N) candidates");
        for (int it = 0; it < p.iters; ++it) {
            {
                ProfScope ps("select", 19.0 * L.N, s);
                k_sel_count<<<kSelBlocks, kSelBlock, 0, s>>>(m, it);
                BP_LAUNCH();
                k_sel_apply<<<kSelBlocks, kSelBlock, 0, s>>>(m, ties);
                BP_LAUNCH();
                k_sel_ties<<<kSelBlocks, kSelBlock, 0, s>>>(m, ties, it);
                BP_LAUNCH();
            }
            p.resume = true;
            p.pending = it + 1 == p.iters;  // a level that is balanced needs no gains after its last selection
            if (p.pending) break;
            ProfScope ps("move_update", 0.0, s);
            k_move_pairs<<<152 * 8, kBlock, 0, s>>>(m, true);
            BP_LAUNCH();
            k_move_gains<<<152 * 8, kLbBlock, 0, s>>>(m, L.tsn(), warp_sum, true);
            BP_LAUNCH();
        }
    }
    for (int64_t stops = 0;; ++stops) {
        unsigned *slot = p.suspend ? flag_slot(g) : nullptr;
        {
            // every selection streams gain and side twice; the start streams the hyperedges and pins
            ProfScope ps("refine_loop", 10.0 * L.N * std::max(p.iters, 1) + 5.0 * L.N +
                                            (p.start ? 11.0 * L.N + 12.0 * L.E + 5.0 * L.P : 0.0), s);
            launch_refine_loop(s, m, p, cand, dev_status(g), slot);
        }
        if (!p.suspend || !device_flag(g, &ls->pending)) break;
        if (stops > (int64_t)p.iters + L.N + 2) throw Fail{BIPART_ERR_TIMEOUT, "refinement made no progress"};
        ProfScope ps("move_update", 0.0, s);
        k_move_pairs<<<152 * 8, kBlock, 0, s>>>(m, false);
        BP_LAUNCH();
        k_move_gains<<<152 * 8, kLbBlock, 0, s>>>(m, L.tsn(), warp_sum, false);
        BP_LAUNCH();
        p.resume = true;
        p.pending = false;
    }
}

}  // namespace

void uncoarsen(bipart_graph *g, std::vector<Level *> &levels, const int64_t limit[2], int64_t W, int m0,
               int m, int32_t iters, uint8_t *d_side0, int tail_from) {
    cudaStream_t s = g->stream;
    const int Lc = (int)levels.size() - 1;
    const int top = tail_from >= 0 ? tail_from : Lc;  // the coarsest level refined on the grid
    int64_t nmax = 1, emax = 1, ents = 1;
    for (int l = 0; l <= top; ++l) {
        const Level &L = *levels[l];
        nmax = std::max<int64_t>(nmax, L.N);
        emax = std::max<int64_t>(emax, L.E);
        // a node of d incidences takes max(1, ceil(d / run)) <= 1 + d / run entries of the move list
        ents = std::max<int64_t>(ents, L.N + (int64_t)L.P / (short_lists(L) ? kMoveRunShort : kMoveRun));
    }
    Work &w = g->w;
    auto *sa = (uint8_t *)w.side_a.ensure((size_t)nmax, s);
    auto *sb = (uint8_t *)w.side_b.ensure((size_t)nmax, s);
    w.side_prev.ensure((size_t)nmax, s);
    // the coarsening's scratch of the same handle is free by now: at many nodes and few pins these two would be a
    // third of a request's memory
    w.n_c.ensure(sizeof(int) * (size_t)nmax, s);
    w.n_key.ensure(sizeof(int4) * (size_t)ents, s);
    w.pair.ensure(sizeof(unsigned long long) * (size_t)emax, s);
    static_assert(kMoveRunShort == 16 && kMoveRun == 64, "run_shift");
    w.items.ensure(sizeof(int4) * (size_t)kItemCap, s);

    LoopParams p{};
    p.W = W;
    p.limit0 = limit[0];
    p.limit1 = limit[1];
    p.m0 = m0;
    p.m = m;
    p.iters = iters;
    uint8_t *cur = sa, *other = sb;
    // with the tail, the levels from tail_from down are done and sa holds level tail_from's side
    for (int l = top; l >= 0; --l) {
        if (tail_from >= 0 && l == top) continue;
        Level *L = levels[l];
        prof_level('r', l);
        p.initial = l == Lc;
        if (L->N > 0) refine_level(g, *L, p.initial ? nullptr : L->cmap(), cur, p.initial ? 0 : levels[l + 1]->N, p.initial ? cur : other, p);
        if (!p.initial) std::swap(cur, other);
    }
    if (levels[0]->N > 0)
        BP_CUDA(cudaMemcpyAsync(d_side0, cur, (size_t)levels[0]->N, cudaMemcpyDeviceToDevice, s));
}

unsigned *bisect_status_word(bipart_graph *g) { return &loop_state(g)->status0; }

unsigned long long *bisect_weights(bipart_graph *g) { return loop_state(g)->W; }

size_t small_state_bytes() { return 256 + sizeof(LoopState); }

}  // namespace bp
