// Initial partition, refinement and rebalancing of one level in one thread-block-cluster launch
// (Algorithms 3 and 5 and the rebalance of reading C13), with the loops decided on the device.
//
// What bounds it: a round is a short chain of dependent steps (update the gains, histogram, threshold,
// apply, order and move), each far too small for the whole GPU.  As grid launches a round was
// five to eight kernels of 4-25 us plus, outside a captured plan, two host round trips, and every round
// recounted all pins.  Here the steps are separated by cluster barriers (0.5-0.7 us with their L2 round
// trip), the gains are updated from the moved nodes (move_dev.cuh), and every decision is computed by
// every block from the same data, so nothing is read back.  Bisections of the versions before and now:
// 5M x 5M row-net 237 -> 53 ms (600 rebalance rounds: 513 -> 33 us each on the level of 461K nodes and 49M
// pins), 1M-node netlist 3.4 -> 2.8 ms, 90K-node netlist with weighted nets 2.7 -> 1.8 ms.
//
// 512 threads a block: the passes of small levels are bound by the latency of their collectives, which
// 1024 threads made 1.2x slower.  The cluster (one GPC) streams node arrays at a few hundred GB/s; where a
// refinement selection is bound by that the grid takes it (k_sel_count in refine.cu).
//
// Work split: on large levels block r of C owns the node range [r R, (r + 1) R) for the passes over
// nodes (the ranges ascend, so ties are ranked by id from per-block counts); on small ones the
// first block selects alone, with block barriers only.  The warps of all blocks share the move list.
// The counters and histograms that blocks exchange live in L2 (LoopState): every block adds its
// part, and reads the total after the barrier.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstddef>

#include <cooperative_groups.h>
#include <cooperative_groups/scan.h>

#include "common.cuh"
#include "internal.h"
#include "move_dev.cuh"
#include "refine_loop.h"
#include "select_dev.cuh"

namespace bp {

namespace cg = cooperative_groups;

namespace {

struct LoopArgs {
    MoveArgs m;
    unsigned long long *cand;  // rebalance candidates (sq entries): gain descending << 32 | node
    long long W, limit0, limit1, sq, max_rounds;
    int m0, mt;                // Algorithm 3: side 0 grows to m0 / mt of the weight
    int iters;
    bool initial, resume, pending, suspend, solo;
    bool start;                // project the sides and count the gains first (small levels)
    const int *cmap;           // start: node -> node of the coarser level (null: all nodes on side 1)
    const uint8_t *coarse;
    unsigned *pending_slot;    // check slot of the pending flag in a captured plan (or null)
    uint32_t *status;
};

constexpr int kT = kLoopThreads;
constexpr int kWarps = kT / 32;
constexpr int kWinWords = 4096;          // tie bitmap: one window of 131,072 nodes
constexpr int kWin = 32 * kWinWords;
constexpr int kListCap = 4096;           // candidates a block keeps from its pass over the nodes
constexpr int kStep = 8 * kT;            // nodes a block visits between two flushes of the chosen
constexpr int kChosenCap = kStep + 4096;
constexpr int kScan = 4 * kStep;         // nodes a block looks through at once for the few above a guess
constexpr int kHubs = 192;               // chosen nodes of a flush's pass whose long entry lists a warp each writes
constexpr int kFlush = 4;                // nodes a thread in a flush's pass

// The block's view of a launch.  Solo: this block selects for the whole level (the other blocks of the
// cluster only help with the gain updates).
struct Ctx {
    int r, C, lo, hi;
    bool solo;
    bool wvec;                   // the weights are aligned for 16-byte loads (the other node arrays are)
    int p;                       // LoopRound of the last selection
};

// What the threshold leaves to decide: a group's mode and threshold gain, and whether some of its ties stay.
struct Taken {
    unsigned mode[2], thr[2];
    bool some[2], hit;
    // 2: taken, 1: a tie to be ranked, 0: not taken
    __device__ __forceinline__ int operator()(int grp, int g) const {
        const unsigned k = gkey(g), md = grp ? mode[1] : mode[0], th = grp ? thr[1] : thr[0];
        if (md == 1) return 2;
        if (md != 2 || k < th) return 0;
        if (k > th) return 2;
        if (hit) return 0;  // in the bitmap already
        return (grp ? some[1] : some[0]) ? 1 : 2;
    }
};

// Everything the phases share, the launch's arguments among it: they are functions of their own with plain
// arguments, since what is passed by value or reference goes through each thread's stack.
struct Shared {
    LoopArgs a;
    Ctx x;
    unsigned long long inc, weight;  // of the selection at hand (LoopRound)
    int guessed, guess;          // rebalance: the last round's threshold gain, if there is one
    LoopRound rd;                // solo: the round's counters
    alignas(16) RState st;       // this block's copy of the selection state; st.hist: its histogram
    unsigned red[32];
    int2 chosen[kChosenCap];     // nodes taken and the side they move to (rebalance candidates: their gain)
    unsigned nlist, nchosen, nhub, base;
    alignas(16) int4 hub[kHubs];  // node, side, first incidence, incidences
    unsigned hub_at[kHubs];
    unsigned ntie[2];
    FindScratch find;
    Taken taken;
    CutScratch cut;
    // the rebalance's sort keys take the place of what follows (and may reach past it)
    alignas(16) unsigned bits[2][kWinWords];  // the threshold's ties per group, one bit per node of the window
    int2 list[kListCap];         // candidates (node | group << 31, gain)
    __device__ unsigned long long *keys() { return reinterpret_cast<unsigned long long *>(&bits[0][0]); }
};

static_assert(offsetof(Shared, st) % 16 == 0 && offsetof(RState, hist) % 16 == 0, "the histogram is read in 16-byte pieces");
static_assert(offsetof(Shared, hub) % 16 == 0, "16-byte entries");
static_assert(offsetof(Shared, bits) % 16 == 0 && offsetof(LoopState, hist) == 0, "aligned");

// The block's shared memory, named so that the compiler sees the address space.
__device__ __forceinline__ Shared &sh() {
    extern __shared__ __align__(16) char smem[];
    return *reinterpret_cast<Shared *>(smem);
}

__device__ __forceinline__ void cluster_sync() {  // all blocks of the cluster
    if (sh().x.C == 1) __syncthreads();
    else cg::this_cluster().sync();
}
__device__ __forceinline__ void sel_sync() {  // the selecting blocks
    if (sh().x.solo) __syncthreads();
    else cluster_sync();
}
__device__ __forceinline__ LoopRound *global_round() { return &sh().a.m.ls->rd[sh().x.p]; }
// A counter of the round, after a barrier of the selecting blocks.
template <class T>
__device__ __forceinline__ T round_count(T LoopRound::*f) {
    return sh().x.solo ? sh().rd.*f : __ldcg(&(global_round()->*f));
}

// A step's eight nodes of a thread: two quads of consecutive nodes; slots of nodes that do not exist
// hold the lowest gain.
struct Step {
    int g[8], w[8];
    unsigned sd[2];
    int v0;
    __device__ __forceinline__ int node(int q) const { return v0 + 4 * ((int)threadIdx.x + (q >> 2) * kT) + (q & 3); }
    __device__ __forceinline__ int side(int q) const { return (int)(sd[q >> 2] >> (8 * (q & 3)) & 255u); }
};

// fn(step) for the nodes [lo, hi) of the block, kStep nodes per step, by all threads, converged.  The gains
// are loaded first, then the sides and weights of the quads that have a node of at least `floor`.  The quad
// at the end of a range is loaded whole (the arrays have slack).
template <class Fn>
__device__ __forceinline__ void visit_nodes(int lo, int hi, int floor, bool need_w,
                                            const uint8_t *sides, Fn fn) {
    const int *gain = sh().a.m.gain, *nw = sh().a.m.nw;
#pragma unroll 1
    for (int v0 = lo; v0 < hi; v0 += kStep) {
        Step t;
        t.v0 = v0;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int v = t.node(4 * u);
            int4 g = make_int4(INT_MIN, INT_MIN, INT_MIN, INT_MIN);
            if (v < hi) g = __ldcg(reinterpret_cast<const int4 *>(gain + v));
            t.g[4 * u] = g.x;
            t.g[4 * u + 1] = v + 1 < hi ? g.y : INT_MIN;
            t.g[4 * u + 2] = v + 2 < hi ? g.z : INT_MIN;
            t.g[4 * u + 3] = v + 3 < hi ? g.w : INT_MIN;
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int v = t.node(4 * u);
            int4 w = make_int4(0, 0, 0, 0);
            t.sd[u] = 0;
            if (max(max(t.g[4 * u], t.g[4 * u + 1]), max(t.g[4 * u + 2], t.g[4 * u + 3])) >= floor) {
                t.sd[u] = __ldcg(reinterpret_cast<const unsigned *>(sides + v));
                if (need_w) {
                    if (sh().x.wvec) w = __ldg(reinterpret_cast<const int4 *>(nw + v));
                    else w = make_int4(__ldg(nw + v), __ldg(nw + v + 1), __ldg(nw + v + 2), __ldg(nw + v + 3));
                }
            }
            t.w[4 * u] = w.x; t.w[4 * u + 1] = w.y; t.w[4 * u + 2] = w.z; t.w[4 * u + 3] = w.w;
        }
        __syncwarp();
        fn(t);
    }
}

// Which nodes a selection may take: gain at least `floor` (and not the lowest value, which no node of
// weight sums below 2^31 has), on side `side` (-1: either), weight at most `room`.
struct Filter {
    int floor, side, room;
    __device__ __forceinline__ bool in(const Step &t, int q) const {
        return t.g[q] >= floor && (side < 0 || t.side(q) == side) && t.w[q] <= room;
    }
};
__device__ __forceinline__ Filter filter(int kind, const RState *st, int floor) {
    return Filter{max(floor, INT_MIN + 1), kind == SEL_REFINE ? -1 : (kind == SEL_INITIAL ? 1 : st->heavy),
                  kind == SEL_REBAL ? (int)min(st->room, (long long)INT_MAX) : INT_MAX};
}

// Places for `n` entries of this lane in a shared list (converged warp; one atomic per warp).
__device__ __forceinline__ unsigned warp_places(unsigned *count, unsigned n) {
    if (__ballot_sync(0xffffffffu, n != 0) == 0) return 0;
    const unsigned inc = warp_inclusive_scan(n);
    unsigned base = 0;
    if ((threadIdx.x & 31) == 31) base = atomicAdd(count, inc);
    return __shfl_sync(0xffffffffu, base, 31) + inc - n;
}

// The chosen nodes join the level's lists: the rebalance's candidates, or (flipped already) the move
// list, one entry per m.run incidences and at least one per node.  All threads.
__device__ __noinline__ void flush_chosen(int kind) {
    Shared &s = sh();
    const MoveArgs &m = s.a.m;
    unsigned inc = 0;
    int weight = 0;
    __syncthreads();
    const int n = (int)s.nchosen;
    if (n == 0) return;  // block-uniform
    if (kind == SEL_REBAL) {
        if (s.x.solo) return;  // at most ceil(sqrt kLoopSoloNodes) of them: they stay in shared memory
        if (threadIdx.x == 0) s.base = atomicAdd(&global_round()->cands, (unsigned)n);
        __syncthreads();
#pragma unroll 1
        for (int i = threadIdx.x; i < n; i += kT)
            s.a.cand[s.base + i] = (unsigned long long)~gkey(s.chosen[i].y) << 32 | (unsigned)s.chosen[i].x;
    } else {
// Bound by the chain of a node's loads, the scan and the lists' atomic: four nodes a thread share them (one a
        // thread, and the hubs one after another with their offsets read again: 3,000 cycles for every 512 nodes,
        // most of a selection that moves tens of thousands).
#pragma unroll 1
        for (int i0 = 0; i0 < n; i0 += kFlush * kT) {
            int v[kFlush], sd[kFlush], b[kFlush], d[kFlush], w[kFlush], c[kFlush], own = 0;
#pragma unroll
            for (int u = 0; u < kFlush; ++u) {
                const int i = i0 + u * kT + (int)threadIdx.x;
                const int2 x = i < n ? s.chosen[i] : make_int2(-1, 0);
                v[u] = x.x;
                sd[u] = x.y;
                b[u] = v[u] >= 0 ? __ldg(m.noff + v[u]) : 0;
                d[u] = v[u] >= 0 ? __ldg(m.noff + v[u] + 1) : 0;
                w[u] = v[u] >= 0 ? __ldg(m.nw + v[u]) : 0;
            }
#pragma unroll
            for (int u = 0; u < kFlush; ++u) {
                d[u] -= b[u];
                inc += (unsigned)d[u];
                weight += sd[u] ? w[u] : -w[u];
                c[u] = v[u] < 0 ? 0 : (d[u] > 0 ? (int)(((unsigned)d[u] + (unsigned)m.run - 1u) >> m.run_shift) : 1);
                own += c[u];
            }
            unsigned tot;
            const unsigned ex = block_scan32<kT>((unsigned)own, s.red, &tot);
            if (threadIdx.x == 0) {
                if (s.x.solo) {
                    s.base = s.rd.ents;
                    s.rd.ents += tot;
                } else {
                    s.base = atomicAdd(&global_round()->ents, tot);
                }
                s.nhub = 0;
            }
            __syncthreads();
            unsigned o = s.base + ex;
#pragma unroll
            for (int u = 0; u < kFlush; ++u) {
                bool mine = c[u] > 0;
                if (c[u] > 8) {
                    const unsigned h = atomicAdd(&s.nhub, 1u);
                    if (h < (unsigned)kHubs) {
                        s.hub[h] = make_int4(v[u], sd[u], b[u], d[u]);
                        s.hub_at[h] = o;
                        mine = false;
                    }
                }
                if (mine)
#pragma unroll 1
                    for (int q = 0; q < c[u]; ++q) m.ent[o + q] = move_entry(v[u], b[u], d[u], q, sd[u], m.run);
                o += (unsigned)c[u];
            }
            __syncthreads();
            const int hubs = (int)min(s.nhub, (unsigned)kHubs);
#pragma unroll 1
            for (int h = threadIdx.x >> 5; h < hubs; h += kWarps) {  // a warp each
                const int4 hub = s.hub[h];
                const int cnt = (int)(((unsigned)hub.w + (unsigned)m.run - 1u) >> m.run_shift);
#pragma unroll 1
                for (int q = threadIdx.x & 31; q < cnt; q += 32)
                    m.ent[s.hub_at[h] + q] = move_entry(hub.x, hub.z, hub.w, q, hub.y, m.run);
            }
            __syncthreads();
        }
    }
    // a block's share of the incidences stays below 2^31, a warp's of one flush as well
    inc = __reduce_add_sync(0xffffffffu, inc);
    weight = __reduce_add_sync(0xffffffffu, weight);
    if ((threadIdx.x & 31) == 0) {
        if (inc) atomicAdd(&s.inc, (unsigned long long)inc);
        if (weight) atomicAdd(&s.weight, (unsigned long long)(long long)weight);
    }
    __syncthreads();
    if (threadIdx.x == 0) s.nchosen = 0;
    __syncthreads();
}

// The round's sums of this block's flushes (thread 0, after a flush) join its counters.
__device__ __forceinline__ void add_sums() {
    Shared &s = sh();
    if (s.x.solo) {
        s.rd.inc += s.inc;
        s.rd.weight += s.weight;
    } else {
        LoopRound *rd = global_round();
        if (s.inc) atomicAdd(&rd->inc, s.inc);
        if (s.weight) atomicAdd(&rd->weight, s.weight);
    }
    s.inc = s.weight = 0;
}

// A node taken by the selection, in place `o` of the chosen: flipped (refinement, initial partition) or a
// candidate (rebalance).
__device__ __forceinline__ void choose(int kind, unsigned o, int v, int side, int g) {
    if (kind != SEL_REBAL) sh().a.m.side[v] = (uint8_t)(side ^ 1);
    sh().chosen[o] = make_int2(v, kind != SEL_REBAL ? side ^ 1 : g);
}

// The block's histogram becomes the selecting blocks' total.
__device__ __noinline__ void sum_hist() {
    __syncthreads();
    if (sh().x.solo) return;
    unsigned *h = &sh().st.hist[0][0], *g = &sh().a.m.ls->hist[0][0];
#pragma unroll 1
    for (int i = threadIdx.x; i < 2 * kHistBins; i += kT)
        if (h[i]) atomicAdd(g + i, h[i]);
    cluster_sync();
#pragma unroll 2
    for (int i = threadIdx.x; i < kHistBins / 2; i += kT)
        reinterpret_cast<uint4 *>(h)[i] = __ldcg(reinterpret_cast<const uint4 *>(g) + i);
    __syncthreads();
}

__device__ __forceinline__ void clear_pass(int words) {
#pragma unroll 1
    for (int i = threadIdx.x; i < kHistBins / 2; i += kT)
        reinterpret_cast<uint4 *>(&sh().st.hist[0][0])[i] = make_uint4(0, 0, 0, 0);
#pragma unroll 1
    for (int i = threadIdx.x; i < words; i += kT) sh().bits[0][i] = sh().bits[1][i] = 0;
    if (threadIdx.x == 0) {
        sh().nlist = 0;
        sh().ntie[0] = sh().ntie[1] = 0;
    }
    __syncthreads();
}

// The ties of group i among the window's bits (first node w0) whose rank by id, `done` of them in the
// windows before, is below `take`.  All threads.
__device__ __noinline__ unsigned take_ties(int kind, int w0, int words, int i, unsigned take, unsigned done) {
    Shared &s = sh();
    const int tie_gain = (int)(s.st.g[i].thr ^ 0x80000000u);
    const int per = (words + kT - 1) / kT, q0 = (int)threadIdx.x * per, q1 = min(q0 + per, words);
    unsigned own = 0;
#pragma unroll 1
    for (int q = q0; q < q1; ++q) own += (unsigned)__popc(s.bits[i][q]);
    unsigned tot;
    const unsigned run = block_scan32<kT>(own, s.red, &tot);
    const unsigned want = min(take - done, tot);  // this window's first `want` ties
#pragma unroll 1
    for (unsigned c0 = 0; c0 < want; c0 += kStep) {
        // a tie's rank is its place in the list
        const unsigned c1 = min(c0 + (unsigned)kStep, want), at = s.nchosen;
        if (run < c1 && run + own > c0) {
            unsigned rank = run;
#pragma unroll 1
            for (int q = q0; q < q1; ++q) {
                unsigned bits = s.bits[i][q];
                while (bits) {
                    const int v = w0 + 32 * q + __ffs(bits) - 1;
                    bits &= bits - 1;
                    if (rank >= c0 && rank < c1) {
                        choose(kind, at + rank - c0, v, i, tie_gain);
                    }
                    ++rank;
                }
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) s.nchosen = at + (c1 - c0);
        __syncthreads();
        if (s.nchosen > (unsigned)(kChosenCap - kStep)) flush_chosen(kind);
        __syncthreads();
    }
    return done + tot;
}

// Sum over the blocks [0, n) of their tie counts of group i (one load per lane, all lanes get it).
__device__ __forceinline__ unsigned sum_ties(int n, int i) {
    const int lane = threadIdx.x & 31;
    return __reduce_add_sync(0xffffffffu, lane < n ? __ldcg(&global_round()->ties[lane][i]) : 0u);
}

// The application when a block's candidates did not fit its list: its nodes read again.  ties: the block's
// ties met are added to ntie, and marked when the range is one window.
__device__ __noinline__ void apply_nodes(int kind, int floor, bool one_win) {
    Shared &s = sh();
    const Ctx &x = s.x;
    const Taken d = s.taken;
    const Filter f = filter(kind, &s.st, floor);
    unsigned n0 = 0, n1 = 0;
    visit_nodes(x.lo, x.hi, f.floor, kind == SEL_REBAL, s.a.m.side, [&](const Step &t) {
        unsigned in = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int grp = t.side(q);
            const int what = f.in(t, q) ? d(grp, t.g[q]) : 0;
            if (what == 2) in |= 1u << q;
            if (what == 1) {
                if (one_win) atomicOr(&s.bits[grp][(t.node(q) - x.lo) >> 5], 1u << ((t.node(q) - x.lo) & 31));
                if (grp) ++n1;
                else ++n0;
            }
        }
        __syncwarp();
        unsigned o = warp_places(&s.nchosen, (unsigned)__popc(in));
        if (in)
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (in >> q & 1u) choose(kind, o++, t.node(q), t.side(q), t.g[q]);
        __syncthreads();
        if (s.nchosen > (unsigned)(kChosenCap - kStep)) flush_chosen(kind);
        __syncthreads();
    });
    n0 = __reduce_add_sync(0xffffffffu, n0);
    n1 = __reduce_add_sync(0xffffffffu, n1);
    if ((threadIdx.x & 31) == 0 && n0) atomicAdd(&s.ntie[0], n0);
    if ((threadIdx.x & 31) == 0 && n1) atomicAdd(&s.ntie[1], n1);
}

// The first `take` ties of group i of a range longer than the bitmap: window by window, the bitmap filled from
// the nodes again, by the sides before this selection (nodes of the other group may have flipped; rebalance
// sides have not changed).
__device__ __noinline__ void take_windows(int kind, int i, unsigned take) {
    Shared &s = sh();
    const Ctx &x = s.x;
    const int thr = (int)(s.st.g[i].thr ^ 0x80000000u);
    Filter f = filter(kind, &s.st, thr);
    f.side = i;
    unsigned done = 0;
    for (int w0 = x.lo; w0 < x.hi && done < take; w0 += kWin) {
        __syncthreads();
        for (int q = threadIdx.x; q < kWinWords; q += kT) s.bits[i][q] = 0;
        __syncthreads();
        visit_nodes(w0, min(x.hi, w0 + kWin), thr, kind == SEL_REBAL, kind == SEL_REBAL ? s.a.m.side : s.a.m.prev,
                    [&](const Step &t) {
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            if (t.g[q] == thr && f.in(t, q))
                                atomicOr(&s.bits[i][(t.node(q) - w0) >> 5], 1u << ((t.node(q) - w0) & 31));
                    });
        __syncthreads();
        done = take_ties(kind, w0, kWinWords, i, take, done);
    }
}

// The exact radix passes for a threshold in a clamped end bucket (rare).
__device__ __noinline__ void exact_threshold(int kind, bool need_w) {
    Shared &s = sh();
    const Ctx &x = s.x;
    RState *st = &s.st;
    unsigned *total = &s.a.m.ls->hist[0][0];
    const Filter f = filter(kind, st, INT_MIN);
    for (int pass = 0; pass < 3; ++pass) {
        if (!x.solo) {
            cluster_sync();  // every block has read the histogram
            if (x.r == 0)
                for (int i = threadIdx.x; i < 2 * kHistBins; i += kT) total[i] = 0;
            cluster_sync();
        }
        __syncthreads();
        for (int i = threadIdx.x; i < 2 * kHistBins; i += kT) (&st->hist[0][0])[i] = 0;
        __syncthreads();
        visit_nodes(x.lo, x.hi, f.floor, need_w, s.a.m.side, [&](const Step &t) {
#pragma unroll 1
            for (int i = 0; i < 2; ++i) {
                const SelGroup &G = st->g[i];
                if (G.mode != 3 || (f.side >= 0 && f.side != i)) continue;
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const unsigned k = gkey(t.g[q]);
                    if (f.in(t, q) && t.side(q) == i && (kind != SEL_REFINE || t.g[q] >= 0) && k >= G.base &&
                        (unsigned long long)k < G.top)
                        atomicAdd(&st->hist[i][(k - G.base) >> G.shift], 1u);
                }
            }
        });
        sum_hist();
        d_sel_find_exact(st, s.a.status, st->hist);
        __syncthreads();
    }
}

// select_nodes' pass of a rebalance round that starts from a guess, on blocks of more than one step: the ties at
// the guess go into the bitmap (their number is returned), the nodes above it into the histogram and the
// list.  Gains and sides of 32 nodes a thread are in flight, then the weights where one of four is on the
// heavy side and high enough; visit_nodes, with eight and a third load behind the sides, took 2,800 cycles for every
// 4,096 nodes of a block (round on 461K nodes: 21 thousand cycles of 83, now 11 with the wait for the slowest block).
__device__ __noinline__ unsigned scan_guess(int gv, int heavy, int room) {
    Shared &s = sh();
    constexpr int kQ = kScan / (4 * kT);  // quads of consecutive nodes a thread
    const int lo = s.x.lo, hi = s.x.hi;
    const int *gain = s.a.m.gain, *nw = s.a.m.nw;
    const uint8_t *side = s.a.m.side;
    const unsigned want = heavy ? 0x01010101u : 0u;
    const bool wvec = s.x.wvec;
    unsigned mine = 0;
#pragma unroll 1
    for (int v0 = lo; v0 < hi; v0 += kScan) {
        int4 g[kQ], w[kQ];
        unsigned in = 0;  // four bits a quad
#pragma unroll
        for (int k = 0; k < kQ; ++k) {
            const unsigned v = (unsigned)v0 + 4u * (threadIdx.x + (unsigned)(k * kT));
            g[k] = make_int4(INT_MIN, INT_MIN, INT_MIN, INT_MIN);
            w[k].x = (int)~want;  // the sides, until the weights are here
            if (v < (unsigned)hi) {
                g[k] = __ldcg(reinterpret_cast<const int4 *>(gain + v));
                w[k].x = (int)__ldcg(reinterpret_cast<const unsigned *>(side + v));
            }
        }
#pragma unroll
        for (int k = 0; k < kQ; ++k) {
            const int v = v0 + 4 * ((int)threadIdx.x + k * kT);
            const unsigned off = (unsigned)w[k].x ^ want;  // a zero byte: on the side
            if (g[k].x >= gv && (off & 0xffu) == 0) in |= 1u << (4 * k);
            if (g[k].y >= gv && (off & 0xff00u) == 0 && v + 1 < hi) in |= 2u << (4 * k);
            if (g[k].z >= gv && (off & 0xff0000u) == 0 && v + 2 < hi) in |= 4u << (4 * k);
            if (g[k].w >= gv && (off & 0xff000000u) == 0 && v + 3 < hi) in |= 8u << (4 * k);
            w[k] = make_int4(0, 0, 0, 0);
            if (in >> (4 * k) & 15u) {
                if (wvec) w[k] = __ldg(reinterpret_cast<const int4 *>(nw + v));
                else w[k] = make_int4(__ldg(nw + v), __ldg(nw + v + 1), __ldg(nw + v + 2), __ldg(nw + v + 3));
            }
        }
        if (!__any_sync(0xffffffffu, in != 0)) continue;
#pragma unroll
        for (int k = 0; k < kQ; ++k) {
            if (!__any_sync(0xffffffffu, (in >> (4 * k) & 15u) != 0)) continue;
            const int v = v0 + 4 * ((int)threadIdx.x + k * kT);
            unsigned q = in >> (4 * k) & 15u;
            if (w[k].x > room) q &= ~1u;
            if (w[k].y > room) q &= ~2u;
            if (w[k].z > room) q &= ~4u;
            if (w[k].w > room) q &= ~8u;
            const unsigned tie = q & ((g[k].x == gv ? 1u : 0u) | (g[k].y == gv ? 2u : 0u) | (g[k].z == gv ? 4u : 0u) | (g[k].w == gv ? 8u : 0u));
            if (tie) {
                mine += (unsigned)__popc(tie);
                atomicOr(&s.bits[heavy][(v - lo) >> 5], tie << ((v - lo) & 31));
            }
            q &= ~tie;
            if (!__any_sync(0xffffffffu, q != 0)) continue;
            unsigned o = warp_places(&s.nlist, (unsigned)__popc(q));
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int x = c == 0 ? g[k].x : (c == 1 ? g[k].y : (c == 2 ? g[k].z : g[k].w));
                if (q >> c & 1u) {
                    int b = x - kClampLo;
                    b = b < 0 ? 0 : (b > kHistBins - 1 ? kHistBins - 1 : b);
                    atomicAdd(&s.st.hist[heavy][b], 1u);
                    if (o < (unsigned)kListCap) s.list[o] = make_int2((v + c) | (int)((unsigned)heavy << 31), x);
                    ++o;
                }
            }
        }
        __syncwarp();
    }
    return mine;
}

// One selection of Algorithm 3 (SEL_INITIAL), Algorithm 5 (SEL_REFINE) or the rebalance (SEL_REBAL)
// and its application, by the selecting blocks.  The histogram and the lists of x.p ^ 1 are clear.
//
// One pass over the nodes counts the candidates' gains and keeps the candidates (up to kListCap a block)
// for the application, which otherwise reads the nodes again.  Rebalance rounds after a level's first
// start from the last round's threshold gain: nodes below it are not looked at, those at it go
// straight into the tie bitmap, and only when too few are left does the pass start over.
__device__ __noinline__ void select_nodes(int kind) {
    Shared &s = sh();
    const Ctx &x = s.x;
    const LoopArgs &a = s.a;
    RState *st = &s.st;
    const int lo = x.lo, hi = x.hi;
    const bool one_win = hi - lo <= kWin;
    const bool need_w = kind == SEL_REBAL;
    const int words = one_win ? (hi - lo + 31) >> 5 : kWinWords;
    const int heavy = st->heavy, gv = s.guess;
    bool guess = kind == SEL_REBAL && s.guessed && (long long)a.m.N <= (long long)kWin * (x.solo ? 1 : x.C);
    for (;;) {
        const Filter f = filter(kind, st, kind == SEL_REFINE ? 0 : (guess ? gv : INT_MIN));
        clear_pass(one_win ? words : 0);
        unsigned mine = 0;  // ties met
        if (guess && hi - lo > kStep) mine = scan_guess(gv, heavy, f.room);
        else
        visit_nodes(lo, hi, f.floor, need_w, a.m.side, [&](const Step &t) {
            unsigned cand = 0, at = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const bool in = f.in(t, q), tie = guess && t.g[q] == gv;
                if (in && tie) at |= 1u << q;
                if (in && !tie) {
                    cand |= 1u << q;
                    int b = t.g[q] - kClampLo;
                    b = b < 0 ? 0 : (b > kHistBins - 1 ? kHistBins - 1 : b);
                    atomicAdd(&st->hist[f.side < 0 ? t.side(q) : f.side][b], 1u);
                }
            }
            if (at) {
                mine += (unsigned)__popc(at);
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int o = t.node(4 * u) - lo;
                    if (at >> (4 * u) & 15u) atomicOr(&s.bits[heavy][o >> 5], (at >> (4 * u) & 15u) << (o & 31));
                }
            }
            if (__any_sync(0xffffffffu, *(volatile unsigned *)&s.nlist <= (unsigned)kListCap)) {
                unsigned o = warp_places(&s.nlist, (unsigned)__popc(cand));
                if (cand)
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        if (cand >> q & 1u) {
                            if (o < (unsigned)kListCap)
                                s.list[o] = make_int2(t.node(q) | (int)((unsigned)(f.side < 0 ? t.side(q) : f.side) << 31), t.g[q]);
                            ++o;
                        }
            }
        });
        unsigned ties = 0;
        if (guess) {  // ties at the guess, per block
            mine = __reduce_add_sync(0xffffffffu, mine);
            if ((threadIdx.x & 31) == 0 && mine) atomicAdd(&s.ntie[heavy], mine);
            __syncthreads();
            if (threadIdx.x == 0 && !x.solo) global_round()->ties[x.r][heavy] = s.ntie[heavy];
        }
        sum_hist();
        if (guess) ties = x.solo ? s.ntie[heavy] : sum_ties(x.C, heavy);
        if (find_threshold<kT>(st, s.find, kind, a.sq, guess, gv, ties)) break;
        guess = false;
        if (!x.solo) {  // start over: the shared histogram is cleared between two barriers
            cluster_sync();
            if (x.r == 0)
                for (int i = threadIdx.x; i < 2 * kHistBins; i += kT) (&a.m.ls->hist[0][0])[i] = 0;
            cluster_sync();
        }
        __syncthreads();
    }
    const bool hit = s.find.hit != 0;  // the threshold is the guess: its ties are in the bitmap and counted
    const bool slow = s.find.slow != 0;
    if (slow) exact_threshold(kind, need_w);
    Taken d;
    d.hit = hit;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        d.mode[i] = st->g[i].mode;
        d.thr[i] = st->g[i].thr;
        d.some[i] = d.mode[i] == 2 &&
                    (slow || hit || st->hist[i][(int)(d.thr[i] ^ 0x80000000u) - kClampLo] > st->g[i].take_eq);
    }
    if (threadIdx.x == 0) {
        s.nchosen = 0;
        s.taken = d;
    }
    if (guess && !hit) {  // the threshold lies above the guess: its ties come from the list
#pragma unroll 1
        for (int q = threadIdx.x; q < words; q += kT) s.bits[0][q] = s.bits[1][q] = 0;
        if (threadIdx.x < 2) s.ntie[threadIdx.x] = 0;
    }
    __syncthreads();
    if (s.nlist <= (unsigned)kListCap) {
        const int n = (int)s.nlist;
#pragma unroll 1
        for (int i0 = 0; i0 < n; i0 += kT) {
            const int i = i0 + (int)threadIdx.x;
            const int2 c = i < n ? s.list[i] : make_int2(0, 0);
            const int v = c.x & 0x7fffffff, grp = (int)((unsigned)c.x >> 31);
            const int what = i < n ? d(grp, c.y) : 0;
            if (what == 1) {
                if (one_win) atomicOr(&s.bits[grp][(v - lo) >> 5], 1u << ((v - lo) & 31));
                atomicAdd(&s.ntie[grp], 1u);
            }
            __syncwarp();
            const unsigned o = warp_places(&s.nchosen, what == 2);
            if (what == 2) choose(kind, o, v, grp, c.y);
        }
    } else {
        apply_nodes(kind, kind == SEL_REFINE ? 0 : (guess ? gv + 1 : INT_MIN), one_win);
    }
    if (d.some[0] || d.some[1]) {  // the same in every block
        __syncthreads();
        if (!x.solo && !hit) {
            if (threadIdx.x < 2) global_round()->ties[x.r][threadIdx.x] = s.ntie[threadIdx.x];
            cluster_sync();
        }
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {
            if (!(i ? d.some[1] : d.some[0])) continue;
            // ties are taken by ascending id: the blocks before this one take theirs first
            const unsigned want = st->g[i].take_eq, before = x.solo ? 0u : sum_ties(x.r, i);
            const unsigned take = before >= want ? 0u : min(s.ntie[i], want - before);
            if (take == 0) continue;  // block-uniform
            if (one_win) take_ties(kind, lo, words, i, take, 0);
            else take_windows(kind, i, take);
        }
    }
    flush_chosen(kind);
    if (threadIdx.x == 0) {
        const int i = heavy > 0;
        s.guessed = kind == SEL_REBAL && heavy >= 0 && !slow && d.mode[i] == 2;
        s.guess = (int)((i ? d.thr[1] : d.thr[0]) ^ 0x80000000u);
    }
    if (kind != SEL_REBAL && threadIdx.x == 0) add_sums();
    sel_sync();
}

// The level's pairs and gains counted from the sides (what k_hedge_n1 and k_node_gain do on large levels), by all
// blocks, hyperedge by hyperedge: its side-1 pins counted, its pair stored, its contributions added to its pins'
// gains, which are zero.  Up to 32 pins take one thread, more a warp.  Levels whose nodes have many incidences add
// up in shared memory first: few nodes would take many atomics each.
__device__ __noinline__ void count_level() {
    Shared &s = sh();
    const Ctx &x = s.x;
    const MoveArgs &m = s.a.m;
    const int rank = x.r * kT + (int)threadIdx.x, size = x.C * kT, lane = threadIdx.x & 31;
    constexpr int kAcc = (int)(sizeof(s.chosen) / sizeof(int));
    int *acc = reinterpret_cast<int *>(sh().chosen);
    const bool priv = m.N <= kAcc && m.P > 8 * m.N;
    if (priv)
        for (int v = threadIdx.x; v < m.N; v += kT) acc[v] = 0;
    cluster_sync();
    auto add = [&](int v, int c) {
        if (priv) atomicAdd(acc + v, c);
        else atomicAdd(m.gain + v, c);
    };
#pragma unroll 1
    for (int e0 = (rank & ~31); e0 < m.E; e0 += size) {
        const int e = e0 + lane;
        int b = 0, d = 0;
        if (e < m.E) {
            b = __ldg(m.hoff + e);
            d = __ldg(m.hoff + e + 1) - b;
        }
        if (d > 0 && d <= 32) {
            unsigned on1 = 0;
#pragma unroll 4
            for (int i = 0; i < d; ++i) on1 |= (unsigned)__ldcg(m.side + __ldg(m.pins + b + i)) << i;
            const int n1 = __popc(on1), n0 = d - n1, w = m.hw ? __ldg(m.hw + e) : 1;
            m.pair[e] = (unsigned long long)(unsigned)n0 << 32 | (unsigned)n1;
            const int c0 = w * contrib(n0, n1), c1 = w * contrib(n1, n0);
            if (c0 | c1)
#pragma unroll 1
                for (int i = 0; i < d; ++i) {
                    const int c = on1 >> i & 1u ? c1 : c0;
                    if (c) add(__ldg(m.pins + b + i), c);
                }
        }
        unsigned wide = __ballot_sync(0xffffffffu, d > 32);
        while (wide) {
            const int src = __ffs(wide) - 1;
            wide &= wide - 1;
            const int we = e0 + src, wb = __shfl_sync(0xffffffffu, b, src), wd = __shfl_sync(0xffffffffu, d, src);
            int n1 = 0;
#pragma unroll 4
            for (int i = lane; i < wd; i += 32) n1 += (int)__ldcg(m.side + __ldg(m.pins + wb + i));
            n1 = __reduce_add_sync(0xffffffffu, n1);
            const int n0 = wd - n1, w = m.hw ? __ldg(m.hw + we) : 1;
            if (lane == 0) m.pair[we] = (unsigned long long)(unsigned)n0 << 32 | (unsigned)n1;
            const int c0 = w * contrib(n0, n1), c1 = w * contrib(n1, n0);
            if (c0 | c1)
#pragma unroll 1
                for (int i = lane; i < wd; i += 32) {
                    const int v = __ldg(m.pins + wb + i);
                    const int c = __ldcg(m.side + v) ? c1 : c0;
                    if (c) add(v, c);
                }
        }
    }
    if (priv) {
        __syncthreads();
        for (int v = threadIdx.x; v < m.N; v += kT)
            if (acc[v]) atomicAdd(m.gain + v, acc[v]);
    }
    cluster_sync();
}

// The level's sides projected and everything counted, by all blocks (small levels).
__device__ __noinline__ void start_level() {
    const LoopArgs &a = sh().a;
    const MoveArgs &m = a.m;
    const int r = sh().x.r, C = sh().x.C;
#pragma unroll 1
    for (int v = r * kT + (int)threadIdx.x; v < m.N; v += C * kT) {
        const uint8_t sd = a.cmap ? __ldg(a.coarse + __ldg(a.cmap + v)) : (uint8_t)1;
        m.side[v] = sd;
        m.prev[v] = sd;
        m.gain[v] = 0;
    }
    if (r == C - 1)
        for (int i = threadIdx.x; i < (int)(offsetof(LoopState, cmd) / sizeof(unsigned)); i += kT)
            reinterpret_cast<unsigned *>(m.ls)[i] = 0;
    count_level();
}

// Gains after the last selection's moves, by all blocks.  own: exact for the moved nodes too (a
// rebalance leaves them out: they are on the light side, which stays the light side until the
// level is done).
__device__ __noinline__ void update_gains(bool own) {
    Shared &s = sh();
    const Ctx &x = s.x;
    const MoveArgs &m = s.a.m;
    LoopState *ls = m.ls;
    const uint8_t *wside = own ? m.prev : m.side;
    const int tid = (int)threadIdx.x;
    unsigned n;
    if (x.solo && x.r == 0) {
        n = s.rd.ents;
        if (x.C == 1 || n <= (unsigned)(2 * kWarps * (32 / m.lanes))) {
            // a short list: this block alone is as fast as the cluster, without its barriers
            move_pass1(m, n, &s.rd.items, tid >> 5, kWarps, wside, false);
            __syncthreads();
            if (own || s.rd.items > 0) {
                move_pass2(m, n, s.rd.items, tid >> 5, kWarps, wside, own);
                __syncthreads();
            }
            if (own) move_settle(m, n, tid, kT);
            if (tid < (int)(sizeof(LoopRound) / sizeof(unsigned))) reinterpret_cast<unsigned *>(&s.rd)[tid] = 0;
            __syncthreads();
            return;
        }
        if (tid == 0) {
            ls->rd[0].ents = n;
            ls->rd[0].items = 0;
            ls->rd[0].inc = s.rd.inc;
            ls->cmd = 1u | (unsigned)own << 1;
        }
        cluster_sync();  // the helpers read the command after this barrier
    } else {
        n = __ldcg(&ls->rd[x.p].ents);
    }
    const bool full = x.solo && (long long)__ldcg(&ls->rd[0].inc) * kMoveCount > (long long)m.P;
    LoopRound *rd = &ls->rd[x.solo ? 0 : x.p];
    // the histogram and the other round's lists are clear for the next selection
    if (!x.solo && x.r == x.C - 1) {
        for (int i = tid; i < 2 * kHistBins; i += kT) (&ls->hist[0][0])[i] = 0;
        unsigned *other = reinterpret_cast<unsigned *>(&ls->rd[x.p ^ 1]);
        for (int i = tid; i < (int)(sizeof(LoopRound) / sizeof(unsigned)); i += kT) other[i] = 0;
    }
    if (full) {
        for (int v = x.r * kT + tid; v < m.N; v += x.C * kT) m.gain[v] = 0;
        count_level();
    } else {
        // a warp per entry, the blocks' first warps first: a short list spreads over all SMs
        const int warp = (tid >> 5) * x.C + x.r, warps = x.C * kWarps;
        move_pass1(m, n, &rd->items, warp, warps, wside, false);
        cluster_sync();
        const unsigned items = __ldcg(&rd->items);
        if (own || items > 0) {
            move_pass2(m, n, items, warp, warps, wside, own);
            cluster_sync();
        }
    }
    if (x.solo) {
        if (x.r != 0) return;
        if (own) move_settle(m, n, tid, kT);
        if (tid < (int)(sizeof(LoopRound) / sizeof(unsigned))) reinterpret_cast<unsigned *>(&s.rd)[tid] = 0;
        __syncthreads();
    } else if (own) {
        move_settle(m, n, x.r * kT + tid, x.C * kT);
    }
}

// Ordered move of the rebalance (reading C13), alike in every selecting block; block r moves every
// C-th node of the prefix.
__device__ __noinline__ void rebal_move() {
    Shared &s = sh();
    const Ctx &x = s.x;
    const LoopArgs &a = s.a;
    unsigned long long *keys = s.keys();
    RState *st = &s.st;
    const int n = x.solo ? (int)s.nchosen : (int)__ldcg(&global_round()->cands);
    if (n == 0) {
        __syncthreads();
        if (threadIdx.x == 0) st->warn = 1;
        sel_sync();
        return;
    }
    const int heavy = st->heavy;
    int S = 1;
    while (S < n) S <<= 1;
    unsigned total = 0;
#pragma unroll 1
    for (int i = threadIdx.x; i < S; i += kT) {
        unsigned long long k = ~0ull;
        if (i < n) {
            k = x.solo ? (unsigned long long)~gkey(s.chosen[i].y) << 32 | (unsigned)s.chosen[i].x : __ldcg(a.cand + i);
            total += (unsigned)__ldg(a.m.nw + (unsigned)k);
        }
        keys[i] = k;
    }
    total = block_sum32<kT>(total, s.red);
    unsigned moved;
    const int cut = rebal_prefix<kT>(keys, n, a.sq, st->room, st->need, a.m.nw, total, s.red, s.cut, &moved);
    if (threadIdx.x == 0) {
        st->W[1 - heavy] += moved;
        st->W[heavy] -= moved;
    }
    __syncthreads();
    const int D = x.solo ? 1 : x.C, r = x.solo ? 0 : x.r;
    for (int b0 = 0; b0 < cut; b0 += kStep * D) {
        const int left = min(cut - b0 - r + D - 1, kStep * D) / D;  // this block's nodes of the step
        for (int i = threadIdx.x; i < left; i += kT) {
            const int v = (int)(unsigned)keys[b0 + i * D + r];
            a.m.side[v] = (uint8_t)(1 - heavy);
            s.chosen[i] = make_int2(v, 1 - heavy);
        }
        if (threadIdx.x == 0) s.nchosen = (unsigned)max(left, 0);
        flush_chosen(SEL_REFINE);
    }
    if (threadIdx.x == 0) add_sums();
    sel_sync();
}

// The side weights after a selection's moves (one thread).
__device__ __forceinline__ void move_weight() {
    RState &st = sh().st;
    const unsigned long long w = round_count(&LoopRound::weight);
    st.W[1] += w;
    st.W[0] -= w;
}

__device__ __forceinline__ bool too_large() {
    return sh().a.suspend && round_count(&LoopRound::inc) > (unsigned long long)kLoopMoveInc;
}

// End of the launch for the selecting blocks (solo: the helpers are sent home).
__device__ __noinline__ void leave(unsigned pending, int it, bool rebal) {
    const LoopArgs &a = sh().a;
    const Ctx &x = sh().x;
    LoopState *ls = a.m.ls;
    if (x.r == 0 && threadIdx.x == 0) {
        const RState &st = sh().st;
        ls->cmd = 0;
        ls->pending = pending;
        if (x.solo) {
            ls->rd[0] = sh().rd;
            ls->rd[0].items = 0;
        }
        ls->sel = x.solo ? 0u : (unsigned)x.p;
        ls->it = (unsigned)it;
        ls->status0 = st.warn;
        ls->rebal = rebal;
        ls->rounds = st.rounds;
        ls->heavy = st.heavy;
        ls->W[0] = st.W[0];
        ls->W[1] = st.W[1];
        ls->room = st.room;
        ls->need = st.need;
        if (a.pending_slot) *a.pending_slot = pending;
    }
    if (x.solo && x.C > 1) cluster_sync();
}

}  // namespace

__global__ void __launch_bounds__(kLoopThreads, 1) k_refine_loop(const __grid_constant__ LoopArgs args) {
    Shared &s = sh();
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), r = (int)cl.block_rank();
    for (int i = threadIdx.x; i < (int)(sizeof(LoopArgs) / sizeof(int)); i += kT)
        reinterpret_cast<int *>(&s.a)[i] = reinterpret_cast<const int *>(&args)[i];
    if (threadIdx.x < sizeof(LoopRound) / sizeof(unsigned)) reinterpret_cast<unsigned *>(&s.rd)[threadIdx.x] = 0;
    RState *st = &s.st;
    LoopState *ls = args.m.ls;
    if (threadIdx.x == 0) {
        const int parts = args.solo ? 1 : C;
        const int R = (int)(((long long)args.m.N + parts - 1) / parts + 31) & ~31;
        s.x.r = r;
        s.x.C = C;
        s.x.lo = args.solo ? 0 : (int)min((long long)R * r, (long long)args.m.N);
        s.x.hi = (int)min((long long)s.x.lo + R, (long long)args.m.N);
        s.x.solo = args.solo;
        s.x.wvec = (reinterpret_cast<uintptr_t>(args.m.nw) & 15) == 0;
        s.x.p = args.resume ? (int)__ldcg(&ls->sel) : 1;
        s.guessed = 0;
        s.inc = s.weight = 0;
        s.nchosen = 0;
        st->heavy = -1;
        st->warn = 0;
        st->rounds = 0;
        st->slow = 0;
        st->flag = 0;
        st->room = st->need = 0;
        // the side weights as the coarser level (or the stop) left them
        st->W[0] = __ldcg(&ls->W[0]);
        st->W[1] = __ldcg(&ls->W[1]);
    }
    __syncthreads();
    const LoopArgs &a = s.a;
    const bool pend = a.resume && a.pending && __ldcg(&ls->go) != 0;
    if (a.resume && !pend) {
        move_settle(a.m, __ldcg(&global_round()->ents), r * kT + (int)threadIdx.x, C * kT);
        if (a.solo) cluster_sync();
    }
    if (a.start && !a.resume) start_level();
    if (a.solo && r != 0) {  // helper: gain updates as the first block commands
        if (threadIdx.x == 0) s.x.p = 0;
        for (;;) {
            cluster_sync();
            const unsigned cmd = __ldcg(&ls->cmd);
            if (cmd == 0) return;
            update_gains((cmd & 2u) != 0);
        }
    }
    int it = 0;
    bool pending = pend;    // the last selection's moves are not in the gains yet
    bool in_rebal = false;
    auto select = [&](int kind) {
        __syncthreads();
        if (threadIdx.x == 0) s.x.p ^= 1;
        __syncthreads();
        select_nodes(kind);
        pending = true;
    };
    if (a.resume) {
        it = (int)__ldcg(&ls->it);
        in_rebal = __ldcg(&ls->rebal) != 0;
        if (threadIdx.x == 0 && in_rebal) {
            st->rounds = __ldcg(&ls->rounds);
            st->heavy = __ldcg(&ls->heavy);
            st->room = __ldcg(&ls->room);
            st->need = __ldcg(&ls->need);
            st->flag = 1;
        }
        __syncthreads();
    }
    // Algorithm 3, then Algorithm 5's iterations, then the rebalance: one loop, so that its phases are one copy
    // of the code
    int kind = a.initial && !a.resume ? SEL_INITIAL : (in_rebal ? SEL_REBAL : SEL_REFINE);
    bool first = !in_rebal;  // the loop condition of this kind is evaluated for the first time
    bool own = !in_rebal;    // the rebalance's first update covers the refinement's moves, exact for every node
    if (kind == SEL_INITIAL && threadIdx.x == 0) {
        st->W[0] = 0;
        st->W[1] = (unsigned long long)a.W;
    }
    for (;;) {
        // the conditions of the loops: Algorithm 3's share, the iteration count, the balance limit
        if (!(in_rebal && first == false && kind == SEL_REBAL && st->flag && !pending)) {
            if (threadIdx.x == 0) {
                if (kind == SEL_INITIAL) d_initial_cond(st, a.max_rounds, a.status, first, a.m0, a.mt);
                else if (kind == SEL_REFINE) st->flag = it < a.iters;
                else d_rebal_cond(st, a.limit0, a.limit1, a.max_rounds, a.status, first);
            }
            __syncthreads();
        }
        first = false;
        if (!st->flag) {
            __syncthreads();
            if (kind == SEL_REBAL) break;
            kind = kind == SEL_INITIAL ? SEL_REFINE : SEL_REBAL;
            first = true;
            continue;
        }
        if (pending) {
            if (kind != SEL_INITIAL && too_large()) {
                leave(1, it, kind == SEL_REBAL && !own);
                return;
            }
            update_gains(kind != SEL_REBAL || own);
            if (kind == SEL_REBAL) own = false;
        }
        select(kind);
        if (kind == SEL_REBAL) {
            own = false;
            rebal_move();
        } else if (threadIdx.x == 0) {
            move_weight();
        }
        if (kind == SEL_REFINE) ++it;
        in_rebal = false;
    }
    leave(0, it, false);
}

// ------------------------------------------------------------------------ host side
namespace {
constexpr size_t kLoopKeys = sizeof(Shared) - offsetof(Shared, bits);  // bytes the sort keys have without asking

// Dynamic shared memory of a launch whose rebalance sorts up to sq keys.
size_t loop_smem(int64_t sq) {
    size_t keys = sizeof(unsigned long long);
    while (keys < sizeof(unsigned long long) * (size_t)sq) keys <<= 1;
    return sizeof(Shared) + (keys > kLoopKeys ? keys - kLoopKeys : 0);
}
}  // namespace

// Largest cluster of k_refine_loop the current device runs (1 always works).
static int loop_cluster() {
    static PerDevice cluster;
    return cluster.get([]() {
        BP_CUDA(cudaFuncSetAttribute(k_refine_loop, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)loop_smem(kRebalMax)));
        BP_CUDA(cudaFuncSetAttribute(k_refine_loop, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        for (int c : {kLoopMaxCluster, 8, 4, 2, 1}) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(c);
            cfg.blockDim = dim3(kLoopThreads);
            cfg.dynamicSmemBytes = loop_smem(kRebalMax);
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = c;
            at[0].val.clusterDim.y = 1;
            at[0].val.clusterDim.z = 1;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, k_refine_loop, &cfg) == cudaSuccess && n >= 1) return c;
            cudaGetLastError();
        }
        throw Fail{BIPART_ERR_CUDA, "the refinement kernel does not fit this GPU"};
    });
}

void refine_init() { loop_cluster(); }

void launch_refine_loop(cudaStream_t s, const MoveArgs &m, const LoopParams &p, unsigned long long *cand,
                        uint32_t *status,
                        unsigned *pending_slot) {
    LoopArgs a{};
    a.m = m;
    a.cand = cand;
    a.W = p.W;
    a.limit0 = p.limit0;
    a.limit1 = p.limit1;
    a.sq = p.sq;
    a.max_rounds = (long long)m.N + 1;
    a.m0 = p.m0;
    a.mt = p.m;
    a.iters = p.iters;
    a.initial = p.initial;
    a.resume = p.resume;
    a.pending = p.pending;
    a.suspend = p.suspend;
    a.start = p.start;
    a.cmap = p.cmap;
    a.coarse = p.coarse;
    a.pending_slot = pending_slot;
    a.status = status;
    a.solo = m.N <= kLoopSoloNodes;
    const int C = loop_cluster();
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(kLoopThreads);
    cfg.dynamicSmemBytes = loop_smem(p.sq);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    BP_CUDA(cudaLaunchKernelEx(&cfg, k_refine_loop, a));
    BP_LAUNCH();
}

}  // namespace bp
