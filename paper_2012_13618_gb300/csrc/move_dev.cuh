// Gains kept current under moves (Algorithm 4 without the recount): device code shared by the
// cluster launch that refines a level (refine_loop.cu) and the grid kernels that take its largest
// moves (refine.cu).
//
// Per hyperedge e the pair (n0, n1) counts its pins per side; its contribution to a pin on side i is
// c_i = w ([n_i == 1] - [n_other == 0]), which is Algorithm 4's +w for a pin alone on its side and -w
// for a pin of an uncut hyperedge (a hyperedge of a level has at least two pins, so never both).
// Moving a node changes the pairs of its hyperedges only, and a pair's contributions only where it
// passes the counts 0, 1, d - 1 or d.  So a selection that moved m nodes costs their incidences plus
// the pins of the few hyperedges whose contributions changed, instead of every pin of the level
// (row-net hypergraph of 5M rows: 70-100 thousand incidences a rebalance round against 5-57
// million pins).
//
//   pass 1  every incidence (v, e) of a moved v: the pair of e takes v's move by one 64-bit atomic,
//           whose old value gives that single move's change (x0, x1) of the contributions; where it is
//           not zero, every pin u of e adds x_prev(u), prev = its side before the selection.  The
//           changes of successive moves telescope, so whatever the order of the atomics every gain
//           ends at sum c_prev(u) over the final pairs: exact for the nodes that did not move.
//   pass 2  a moved node's own correction, sum over its hyperedges of c_new - c_prev, and the pins
//           of wide hyperedges queued as work items by pass 1.
//
// All arithmetic is integer addition: the result is the same integers as a full recount.
#pragma once

#include <cooperative_groups.h>

#include "refine_loop.h"

namespace bp {

constexpr int kMoveBatch = 2;    // incidences of an entry a lane takes: an entry's run is 2 * lanes at most
static_assert(kMoveRun == 32 * kMoveBatch && kMoveRunShort == 8 * kMoveBatch, "one batch an entry");
constexpr int kWalkWarp = 512;   // hyperedges up to this degree are walked by the warp that met them, wider ones
constexpr int kWalkShort = 64;   // queued; in short lists up to this one, so that no warp walks many pins

__device__ __forceinline__ int contrib(int own, int other) { return (own == 1) - (other == 0); }

// The pair change of one move to side 1 (s = 1) or side 0.
__device__ __forceinline__ unsigned long long pair_step(int s) {
    return s ? 1ull - (1ull << 32) : (1ull << 32) - 1ull;
}

// Entry q of a moved node's incidence list (first b, length d), `run` a piece, the node now on side s.
__device__ __forceinline__ int4 move_entry(int v, int b, int d, int q, int s, int run) {
    return make_int4(v, b + q * run, b + q * run + min(d - q * run, run), s);
}

// Adds x0 / x1 to the gains of pins [a, b) on side 0 / 1 of `wside`; thread `t` of `nt`.
static __device__ __noinline__ void walk_pins(const int *pins, const uint8_t *wside, int *gain, int a, int b,
                                          int x0, int x1, int t, int nt) {
#pragma unroll 1
    for (int i0 = a + t; i0 < b; i0 += 4 * nt) {
        int u[4], s[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) u[k] = i0 + k * nt < b ? __ldg(pins + i0 + k * nt) : -1;
#pragma unroll
        for (int k = 0; k < 4; ++k) s[k] = u[k] >= 0 ? (int)__ldcg(wside + u[k]) : 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int x = s[k] ? x1 : x0;
            if (u[k] >= 0 && x) atomicAdd(gain + u[k], x);
        }
    }
}

// A wide hyperedge (pins [a, a + d)) whose changes are x0 / x1, queued for pass 2, one place per kItemPins pins.
static __device__ __noinline__ void queue_wide(const MoveArgs &m, unsigned *queued, const uint8_t *wside, int a, int d,
                                               int x0, int x1) {
    const unsigned items = d > 0 ? (unsigned)(d + kItemPins - 1) / kItemPins : 0u;
    const unsigned upto = warp_inclusive_scan(items);
    unsigned base = 0;
    if ((threadIdx.x & 31) == 31) base = atomicAdd(queued, upto);
    base = __shfl_sync(0xffffffffu, base, 31) + upto - items;
#pragma unroll 1
    for (unsigned i = 0; i < items; ++i) {
        const int p0 = a + (int)i * kItemPins, p1 = min(p0 + kItemPins, a + d);
        if (base + i < (unsigned)m.item_cap) m.items[base + i] = make_int4(p0, p1, x0, x1);
        else walk_pins(m.pins, wside, m.gain, p0, p1, x0, x1, 0, 1);  // a full queue
    }
    __syncwarp();
}

// Every lane's two hyperedges (pins [a, a + d), d = 0: none) add their changes x0 / x1 to their pins.  The warp
// walks the pins of all lanes as one sequence, 128 in flight: a lane walking its own hyperedge held the
// others up for the longest one's chain of loads (5M x 5M row-net, level of 461K nodes: pass 1 of a
// rebalance round 25 us with the wait for the slowest warp, now 11).
static __device__ __noinline__ void walk_changed(const MoveArgs &m, const uint8_t *wside, int a, int d, int x0, int x1,
                                                 int b, int f, int z0, int z1) {
    const int lane = threadIdx.x & 31;
    const int upto = (int)warp_inclusive_scan((unsigned)(d + f)), first = upto - d - f;
    const int total = __shfl_sync(0xffffffffu, upto, 31);
#pragma unroll 1
    for (int i0 = 0; i0 < total; i0 += 128) {
        int u[4], s[4], y0[4], y1[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            u[k] = -1;
            y0[k] = y1[k] = 0;
            if (i0 + 32 * k >= total) continue;  // warp-uniform
            const int i = i0 + 32 * k + lane;
            int l = 0;  // the lane pin i belongs to: the last one whose pins start at or before it
#pragma unroll
            for (int h = 16; h > 0; h >>= 1) {
                const int at = __shfl_sync(0xffffffffu, first, l + h);
                if (at <= i) l += h;
            }
            const int o = i - __shfl_sync(0xffffffffu, first, l), da = __shfl_sync(0xffffffffu, d, l);
            const int pa = __shfl_sync(0xffffffffu, a, l), pb = __shfl_sync(0xffffffffu, b, l);
            const int xa0 = __shfl_sync(0xffffffffu, x0, l), xa1 = __shfl_sync(0xffffffffu, x1, l);
            const int xb0 = __shfl_sync(0xffffffffu, z0, l), xb1 = __shfl_sync(0xffffffffu, z1, l);
            y0[k] = o < da ? xa0 : xb0;
            y1[k] = o < da ? xa1 : xb1;
            if (i < total) u[k] = __ldg(m.pins + (o < da ? pa + o : pb + (o - da)));
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) s[k] = u[k] >= 0 ? (int)__ldcg(wside + u[k]) : 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int x = s[k] ? y1[k] : y0[k];
            if (u[k] >= 0 && x) atomicAdd(m.gain + u[k], x);
        }
    }
}

// Pass 1 over the move list's n entries by warps [warp, warps).  queued: the count of work items (zero
// before the pass).  wside: the sides the walked pins are read by (prev, or the current sides when moved
// nodes' gains are not needed any more).  With `full` only the pairs are brought up to date.
static __device__ __noinline__ void move_pass1(const MoveArgs &m, unsigned n, unsigned *queued, int warp, int warps,
                                  const uint8_t *wside, bool full) {
    const int lane = threadIdx.x & 31;
    const int per = 32 / m.lanes, sub = lane % m.lanes, slot = lane / m.lanes;
    // The pass is bound by chains of entry, incidence, atomic, pin and side: a warp has two entries (two incidences
    // a lane each) in flight and the next two loaded ahead.  Offsets are read beside the atomic unless the list
    // is long (then by few lanes of many).
    const bool early = n <= (unsigned)(2 * warps * per), beside = n <= (unsigned)(32 * warps * per);
    const unsigned stride = (unsigned)warps * per, first = (unsigned)warp * per + slot;
    int4 next[2];
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        next[p] = make_int4(0, 0, 0, 0);
        if (first + p * stride < n) next[p] = __ldcg(m.ent + first + p * stride);
    }
#pragma unroll 1
    for (unsigned k0 = (unsigned)warp * per; k0 < n; k0 += 2 * stride) {
        int e[2 * kMoveBatch], a[2 * kMoveBatch], d[2 * kMoveBatch], x0[2 * kMoveBatch], x1[2 * kMoveBatch];
        unsigned long long step[2], o[2 * kMoveBatch];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const int4 en = next[p];
            step[p] = pair_step(en.w);
#pragma unroll
            for (int u = 0; u < kMoveBatch; ++u) {
                const int j = en.y + sub + u * m.lanes;
                e[p * kMoveBatch + u] = j < en.z ? __ldg(m.nadj + j) : -1;
            }
            const unsigned k = k0 + slot + (2 + p) * stride;
            next[p] = make_int4(0, 0, 0, 0);
            if (k < n) next[p] = __ldcg(m.ent + k);
        }
        if (full) {
#pragma unroll
            for (int u = 0; u < 2 * kMoveBatch; ++u)
                if (e[u] >= 0) atomicAdd(m.pair + e[u], step[u / kMoveBatch]);
            continue;
        }
#pragma unroll
        for (int u = 0; u < 2 * kMoveBatch; ++u) {
            a[u] = beside && e[u] >= 0 ? __ldg(m.hoff + e[u]) : 0;
            o[u] = e[u] >= 0 ? atomicAdd(m.pair + e[u], step[u / kMoveBatch]) : 0ull;
        }
#pragma unroll
        for (int u = 0; u < 2 * kMoveBatch; ++u) {
            d[u] = x0[u] = x1[u] = 0;
            if (e[u] < 0) continue;
            const unsigned long long q = o[u] + step[u / kMoveBatch];
            const int o0 = (int)(o[u] >> 32), o1 = (int)(unsigned)o[u], q0 = (int)(q >> 32), q1 = (int)(unsigned)q;
            x0[u] = contrib(q0, q1) - contrib(o0, o1);
            x1[u] = contrib(q1, q0) - contrib(o1, o0);
            if (x0[u] | x1[u]) {
                if (!beside) a[u] = __ldg(m.hoff + e[u]);
                d[u] = o0 + o1;
                const int w = m.hw ? __ldg(m.hw + e[u]) : 1;
                x0[u] *= w;
                x1[u] *= w;
            }
        }
#pragma unroll
        for (int u = 0; u < 2 * kMoveBatch; ++u) {
            const bool wide = d[u] > (early ? kWalkShort : kWalkWarp);
            if (!__any_sync(0xffffffffu, wide)) continue;
            queue_wide(m, queued, wside, a[u], wide ? d[u] : 0, x0[u], x1[u]);
            if (wide) d[u] = 0;
        }
#pragma unroll
        for (int u = 0; u < 2 * kMoveBatch; u += 2)
            if (__any_sync(0xffffffffu, (d[u] | d[u + 1]) != 0))
                walk_changed(m, wside, a[u], d[u], x0[u], x1[u], a[u + 1], d[u + 1], x0[u + 1], x1[u + 1]);
    }
}

// Pass 2: the queued items, and with `own` the moved nodes' corrections.
static __device__ __noinline__ void move_pass2(const MoveArgs &m, unsigned n, unsigned queued, int warp, int warps,
                                  const uint8_t *wside, bool own) {
    const int lane = threadIdx.x & 31;
    const int items = (int)min(queued, (unsigned)m.item_cap);
#pragma unroll 1
    for (int i = warp; i < items; i += warps) {
        const int4 it = __ldcg(m.items + i);
        walk_pins(m.pins, wside, m.gain, it.x, it.y, it.z, it.w, lane, 32);
    }
    if (!own) return;
    const int per = 32 / m.lanes, sub = lane % m.lanes, slot = lane / m.lanes;
    for (unsigned k0 = (unsigned)warp * per; k0 < n; k0 += (unsigned)warps * per) {
        const unsigned k = k0 + slot;
        int acc = 0, v = 0;
        if (k < n) {
            const int4 en = __ldcg(m.ent + k);
            v = en.x;
            const int jb = en.z, s = en.w;
#pragma unroll 4
            for (int j = en.y + sub; j < jb; j += m.lanes) {
                const int e = __ldg(m.nadj + j);
                const unsigned long long q = __ldcg(m.pair + e);
                const int q0 = (int)(q >> 32), q1 = (int)(unsigned)q;
                const int x = s ? contrib(q1, q0) - contrib(q0, q1) : contrib(q0, q1) - contrib(q1, q0);
                if (x) acc += m.hw ? x * __ldg(m.hw + e) : x;
            }
        }
#pragma unroll 1
        for (int o = m.lanes >> 1; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o, m.lanes);
        if (sub == 0 && acc) atomicAdd(m.gain + v, acc);
    }
}

// prev brought up to date for the moved nodes, before the next selection's update.
static __device__ __noinline__ void move_settle(const MoveArgs &m, unsigned n, int rank, int size) {
#pragma unroll 2
    for (unsigned k = (unsigned)rank; k < n; k += (unsigned)size) {
        const int4 en = __ldcg(m.ent + k);
        m.prev[en.x] = (uint8_t)en.w;
    }
}

}  // namespace bp
