// The coarse tail of a bisection run as one thread-block-cluster launch (tail.cu): arguments,
// limits, and the arena layout of the coarse levels it builds, which the host mirrors to expose
// those levels as views.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include "refine_dev.cuh"

namespace bp {

constexpr int kTailThreads = 512;         // threads per block of the cluster
constexpr int kTailNodes = 12288;         // largest level (nodes) the tail can start from
constexpr int64_t kTailMaxPins = 4'000'000;  // ... and pins (its shared-memory chunk table)
// Default start: the first level of at most kTailStartPins pins, or of kTailStartFew on levels of at most kTailFewNodes
// nodes (with more, the one block's selections cost more than the grid's launches: uniform hypergraph of 7,000 nodes
// and 28K pins, replays 642 and 665 us from its second level and its first).  Swept as the start (10K, 25K, 35K, 45K
// pins whatever the nodes), geometric means over 80 netlists, row-nets and uniform hypergraphs of 2,000 to 150,000
// nodes, of the times without a tail in replays and with one of a whole cluster from 70K pins in first calls: first
// calls 0.83, 0.74, 0.72, 0.72, replays 0.81, 0.78, 0.79, 0.80; 10K-node uniform replays 782, 730, 811 us from 25K, 35K,
// 45K; 16-way parts of a 250K-node netlist 12.37, 12.36, 12.47 ms; a mix of 12 graphs on the server 49.4, 48.8, 48.5.
// Above ~35K pins a level no longer fits one block's shared memory beside its nodes, and the refinement's passes go
// back to L2.
constexpr int64_t kTailStartPins = 25'000, kTailStartFew = 35'000;
constexpr int kTailFewNodes = kTailNodes / 2;
constexpr int kTailMaxLevels = 64;        // coarse levels one tail may build
constexpr int kTailMaxCluster = 16;
constexpr int kTailChunk = 2048;          // chunk boundaries of a level every this many pins
constexpr int kTailMaxChunks = 510;       // chunks one block may own (shared-memory table)

// Chunks of a level with P pins: chunk c holds the hyperedges whose first pin lies in
// [c * kTailChunk, (c + 1) * kTailChunk); K = ceil(P / kTailChunk).
__host__ __device__ inline int tail_chunks(int P) { return (P + kTailChunk - 1) / kTailChunk; }

struct TailArgs {
    // the starting level (normalised CSR and node weights; its cmap / matching are written)
    int N, E, P;
    const int *hoff, *pins, *hw, *nw;
    int *cmap, *match;
    int policy, max_new, iters, m0, m;
    long long limit0, limit1;
    char *arena;  // coarse levels, tail_layout() one after another
    size_t arena_cap;
    // scratch: per hyperedge of the starting level (sizes and weights of the matched sets, group
    // representatives, staged offsets and weights of contracted hyperedges, work lists of 2E),
    // per pin (2P: staged coarse pins, then distinct pins of wide hyperedges at fine offsets),
    // per node, the starting level's chunk table and the blocks' compaction totals
    int *e_ssize, *e_sweight;
    unsigned *e_rep;
    int *e_soff, *e_shw, *e_list, *p_stage, *n_grp;
    int *ce0, *cp0;  // chunk table of the starting level (tail_chunks(P) + 1 entries each)
    long long *xchg;
    int *sizes;  // {N', E', P'} of every new level (max_new triples; zero past the last)
    int *info;   // [0] new levels built, [1] MiB of arena a run needed but did not have,
                 // [2] algorithmic KiB the launch moved
    uint8_t *side_out;  // bisection of the starting level
    unsigned *status0;  // whether the starting level's rebalance ran out of candidates
    long long W;        // total node weight
    unsigned long long *W_out;  // the starting level's side weights
    uint32_t *status;
    unsigned long long *trace;  // diagnostics (BIPART_TAIL_TRACE, eager calls): phase time stamps
};

constexpr int kTailTraceMax = 8192;

// Byte offsets of one coarse level's arrays in the arena (64-byte aligned; every array is
// followed by at least 16 bytes of slack so aligned 16-byte loads may run past its end).
struct TailLayout {
    size_t nw, cmap, match, ce, cp, hoff, hw, pins, end;
};

__host__ __device__ inline size_t tail_round(size_t bytes) { return (bytes + 16 + 63) & ~size_t(63); }

__host__ __device__ inline TailLayout tail_layout(size_t base, int N, int E, int P, bool weighted) {
    TailLayout t;
    size_t o = base;
    const size_t n = (size_t)(N > 0 ? N : 1), e = (size_t)(E > 0 ? E : 1), p = (size_t)(P > 0 ? P : 1);
    const size_t k = (size_t)tail_chunks(P) + 1;
    t.nw = o;    o += tail_round(4 * n);
    t.cmap = o;  o += tail_round(4 * n);
    t.match = o; o += tail_round(4 * n);
    t.ce = o;    o += tail_round(4 * k);
    t.cp = o;    o += tail_round(4 * k);
    t.hoff = o;  o += tail_round(4 * ((size_t)E + 1));
    t.hw = o;    if (weighted) o += tail_round(4 * e);
    t.pins = o;  o += tail_round(4 * p);
    t.end = o;
    return t;
}

}  // namespace bp
