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

constexpr int kWalkThread = 32;  // long lists: hyperedges up to this degree are walked by one thread,
constexpr int kWalkWarp = 512;   // up to this one by the warp that met them, wider ones queued
constexpr int kWalkShort = 8;    // short lists: wider ones are all queued, so that no warp walks several

__device__ __forceinline__ int contrib(int own, int other) { return (own == 1) - (other == 0); }

// The pair change of one move to side 1 (s = 1) or side 0.
__device__ __forceinline__ unsigned long long pair_step(int s) {
    return s ? 1ull - (1ull << 32) : (1ull << 32) - 1ull;
}

// Entry q of a moved node's incidence list (first b, length d), the node now on side s.
__device__ __forceinline__ int4 move_entry(int v, int b, int d, int q, int s) {
    return make_int4(v, b + q * kMoveRun, min(b + d, b + (q + 1) * kMoveRun), s);
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

// Pass 1 over the move list's n entries by warps [warp, warps).  queued: the count of work items (zero
// before the pass).  wside: the sides the walked pins are read by (prev, or the current sides when moved
// nodes' gains are not needed any more).  With `full` only the pairs are brought up to date.
static __device__ __noinline__ void move_pass1(const MoveArgs &m, unsigned n, unsigned *queued, int warp, int warps,
                                  const uint8_t *wside, bool full) {
    const int lane = threadIdx.x & 31;
    const int per = 32 / m.lanes, sub = lane % m.lanes, slot = lane / m.lanes;
    // a short list is bound by its chain of loads: the offsets are then read beside the atomic
    const bool early = n <= (unsigned)(2 * warps * per);
    for (unsigned k0 = (unsigned)warp * per; k0 < n; k0 += (unsigned)warps * per) {
        const unsigned k = k0 + slot;
        int j = 0, jb = 0;
        unsigned long long step = 0;
        if (k < n) {
            const int4 en = __ldcg(m.ent + k);
            j = en.y + sub;
            jb = en.z;
            step = pair_step(en.w);
        }
        if (full) {
#pragma unroll 4
            for (; j < jb; j += m.lanes) atomicAdd(m.pair + __ldg(m.nadj + j), step);
            continue;
        }
        while (__any_sync(0xffffffffu, j < jb)) {
            int a = 0, d = 0, x0 = 0, x1 = 0;
            if (j < jb) {
                const int e = __ldg(m.nadj + j);
                if (early) a = __ldg(m.hoff + e);
                const unsigned long long o = atomicAdd(m.pair + e, step), q = o + step;
                const int o0 = (int)(o >> 32), o1 = (int)(unsigned)o, q0 = (int)(q >> 32), q1 = (int)(unsigned)q;
                x0 = contrib(q0, q1) - contrib(o0, o1);
                x1 = contrib(q1, q0) - contrib(o1, o0);
                if (x0 | x1) {
                    if (!early) a = __ldg(m.hoff + e);
                    d = o0 + o1;
                    const int w = m.hw ? __ldg(m.hw + e) : 1;
                    x0 *= w;
                    x1 *= w;
                }
            }
            if (d > 0 && d <= (early ? kWalkShort : kWalkThread)) walk_pins(m.pins, wside, m.gain, a, a + d, x0, x1, 0, 1);
            // wide hyperedges queued for pass 2, one place per kItemPins pins
            const unsigned items = d > (early ? kWalkShort : kWalkWarp) ? (unsigned)(d + kItemPins - 1) / kItemPins : 0u;
            if (__any_sync(0xffffffffu, items != 0)) {
                const unsigned upto = warp_inclusive_scan(items);
                unsigned base = 0;
                if (lane == 31) base = atomicAdd(queued, upto);
                base = __shfl_sync(0xffffffffu, base, 31) + upto - items;
#pragma unroll 1
                for (unsigned i = 0; i < items; ++i) {
                    const int p0 = a + (int)i * kItemPins, p1 = min(p0 + kItemPins, a + d);
                    if (base + i < (unsigned)m.item_cap) m.items[base + i] = make_int4(p0, p1, x0, x1);
                    else walk_pins(m.pins, wside, m.gain, p0, p1, x0, x1, 0, 1);  // a full queue
                }
            }
            unsigned wide = early ? 0u : __ballot_sync(0xffffffffu, d > kWalkThread && d <= kWalkWarp);
            while (wide) {
                const int src = __ffs(wide) - 1;
                wide &= wide - 1;
                const int wa = __shfl_sync(0xffffffffu, a, src), wd = __shfl_sync(0xffffffffu, d, src);
                const int y0 = __shfl_sync(0xffffffffu, x0, src), y1 = __shfl_sync(0xffffffffu, x1, src);
                walk_pins(m.pins, wside, m.gain, wa, wa + wd, y0, y1, lane, 32);
            }
            j += m.lanes;
        }
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
