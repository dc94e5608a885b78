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

namespace bp {

namespace {

template <class T>
T *align16(T *p) {
    return reinterpret_cast<T *>((reinterpret_cast<uintptr_t>(p) + 15) & ~uintptr_t(15));
}

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

__global__ void __launch_bounds__(kBlock) k_move_pairs(MoveArgs m) {
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

__global__ void __launch_bounds__(kLbBlock) k_move_gains(MoveArgs m, const int *__restrict__ ts, bool warp_sum) {
    const LoopRound *rd = &m.ls->rd[m.ls->sel];
    if (move_full(m, rd)) {
        d_node_gain(GridTeam(), m.N, m.P, m.noff, m.nadj, m.pair, m.hw, m.side, m.gain, ts, warp_sum);
        return;
    }
    const int tid = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
    move_pass2(m, __ldcg(&rd->ents), __ldcg(&rd->items), tid >> 5, nt >> 5, m.prev, true);
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

// A level's refinement from the sides in `side` (k_level_start projects them from `coarse`, the
// sides of the next coarser level; null: the coarsest level, with Algorithm 3 first).
void refine_level(bipart_graph *g, Level &L, const int *cmap, const uint8_t *coarse, uint8_t *side, LoopParams p) {
    cudaStream_t s = g->stream;
    Work &w = g->w;
    LoopState *ls = loop_state(g);
    MoveArgs m{};
    m.N = L.N; m.E = L.E; m.P = L.P;
    m.noff = L.noff(); m.nadj = L.nadj(); m.hoff = L.hoff(); m.pins = L.pins(); m.hw = L.hw(); m.nw = L.nw();
    m.side = side;
    m.prev = align16(w.side_prev.as<uint8_t>());
    m.gain = align16(w.gain.as<int>());
    m.pair = w.pair.as<unsigned long long>();
    m.ls = ls;
    m.ent = w.ent.as<int4>();
    m.items = w.items.as<int4>();
    m.item_cap = kItemCap;
    // nodes with short incidence lists share a warp four at a time
    const bool short_lists = (int64_t)L.P <= kMoveRunShort * (int64_t)L.N;
    m.lanes = short_lists ? 8 : 32;
    m.run = short_lists ? kMoveRunShort : kMoveRun;
    m.run_shift = short_lists ? 4 : 6;
    p.sq = ceil_sqrt64(L.N);
    if (p.sq > kRebalMax) throw Fail{BIPART_ERR_OOM, "level too large for the ordered rebalance"};
    auto *cand = (unsigned long long *)w.list.ensure(sizeof(unsigned long long) * (size_t)std::max<int64_t>(p.sq, 1), s);
    const bool warp_sum = (int64_t)L.P > kWarpSumDegree * (int64_t)L.N;
    p.start = L.P <= kLoopStartPins;
    p.cmap = cmap;
    p.coarse = coarse;
    if (!p.start) {
        {
            ProfScope ps("project", 11.0 * L.N + 12.0 * L.E, s);
            k_level_start<<<grid_for(std::max(L.N, L.E)), kBlock, 0, s>>>(L.N, L.E, cmap, coarse, side, m.prev,
                                                                          m.gain, m.hoff, m.pair, ls);
            BP_LAUNCH();
        }
        {
            // hoff, pins, one side byte per pin, one atomic per hyperedge run
            ProfScope ps("hedge_n1", 8.0 * L.E + 5.0 * L.P, s);
            k_hedge_n1<<<lb_grid(L.P), kLbBlock, 0, s>>>(L.E, L.P, L.hoff(), L.pins(), side, m.pair, L.tsh());
            BP_LAUNCH();
        }
        // noff, nadj, 8-byte pair gather per incidence (and a weight where it counts), side, gain
        ProfScope ps("node_gain", 9.0 * L.N + 12.0 * L.P, s);
        k_node_gain<<<lb_grid(L.P), kLbBlock, 0, s>>>(L.N, L.P, L.noff(), L.nadj(), m.pair, L.hw(), side, m.gain,
                                                       L.tsn(), warp_sum);
        BP_LAUNCH();
    }
    p.suspend = L.P > kLoopAlonePins;
    p.resume = false;
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
        k_move_pairs<<<152 * 8, kBlock, 0, s>>>(m);
        BP_LAUNCH();
        k_move_gains<<<152 * 8, kLbBlock, 0, s>>>(m, L.tsn(), warp_sum);
        BP_LAUNCH();
        p.resume = true;
    }
}

}  // namespace

void uncoarsen(bipart_graph *g, std::vector<Level *> &levels, const int64_t limit[2], int64_t W, int m0,
               int m, int32_t iters, uint8_t *d_side0, int tail_from) {
    cudaStream_t s = g->stream;
    const int Lc = (int)levels.size() - 1;
    const int top = tail_from >= 0 ? tail_from : Lc;  // the coarsest level refined on the grid
    int64_t nmax = 1, emax = 1, pmax = 1;
    for (int l = 0; l <= top; ++l) {
        nmax = std::max<int64_t>(nmax, levels[l]->N);
        emax = std::max<int64_t>(emax, levels[l]->E);
        pmax = std::max<int64_t>(pmax, levels[l]->P);
    }
    Work &w = g->w;
    uint8_t *sa = side_buffer(w.side_a, nmax, s);
    uint8_t *sb = side_buffer(w.side_b, nmax, s);
    side_buffer(w.side_prev, nmax, s);
    w.gain.ensure(sizeof(int) * (size_t)nmax + 16, s);
    w.pair.ensure(sizeof(unsigned long long) * (size_t)emax, s);
    static_assert(kMoveRunShort == 16 && kMoveRun == 64, "run_shift");
    // a level with short runs has at most kMoveRunShort incidences a node
    w.ent.ensure(sizeof(int4) * (size_t)(nmax + std::max<int64_t>(pmax / kMoveRun, nmax) + 1), s);
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
        if (L->N > 0) refine_level(g, *L, p.initial ? nullptr : L->cmap(), cur, p.initial ? cur : other, p);
        if (!p.initial) std::swap(cur, other);
    }
    if (levels[0]->N > 0)
        BP_CUDA(cudaMemcpyAsync(d_side0, cur, (size_t)levels[0]->N, cudaMemcpyDeviceToDevice, s));
}

uint8_t *side_buffer(Buf &b, int64_t n, cudaStream_t s) { return align16((uint8_t *)b.ensure((size_t)n + 16, s)); }

unsigned *bisect_status_word(bipart_graph *g) { return &loop_state(g)->status0; }

unsigned long long *bisect_weights(bipart_graph *g) { return loop_state(g)->W; }

size_t small_state_bytes() { return 256 + sizeof(LoopState); }

}  // namespace bp
