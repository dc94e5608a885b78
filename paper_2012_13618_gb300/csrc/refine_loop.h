// The refinement of one level as one thread-block-cluster launch (refine_loop.cu): its state in
// the handle's small scratch, its arguments, and the pieces the grid kernels of a large level's
// gain update share with it (move_dev.cuh).
#pragma once

#include <stdint.h>

#include "refine_dev.cuh"

namespace bp {

constexpr int kLoopThreads = 512;       // threads per block of the cluster
constexpr int kLoopMaxCluster = 16;
// Incidences of a moved node one entry of the move list covers: two a lane, for 32 lanes an entry or 8.  With
// 64 for 8 lanes too a warp went through a node of high degree in four batches while others had none.
constexpr int kMoveRun = 64, kMoveRunShort = 16;
constexpr int kItemPins = 128;          // pins of a wide hyperedge one work item covers (four a lane)
constexpr int kItemCap = 1 << 16;       // work items a pass may queue (beyond: walked on the spot)
// Moves of more than this many incidences are brought into the gains by the whole grid instead of
// the one cluster (levels of more than kLoopAlonePins pins only; smaller ones stay in the cluster).
constexpr long long kLoopMoveInc = 1 << 17;
constexpr int64_t kLoopAlonePins = 1 << 18;
// Levels of at most this many pins are started (sides projected, gains counted) by the cluster launch too, unless they
// have more nodes than kLoopStartNodes: its 8,192 threads project a node each at a time.
constexpr int kLoopStartPins = 1 << 17, kLoopStartNodes = 1 << 16;
// Levels of at most this many nodes are selected by the cluster's first block alone, the others helping
// with the gain updates only.
constexpr int kLoopSoloNodes = 4096;
// Above P / kMoveFull moved incidences every gain is recomputed instead of updated; above P / kMoveFullHubs
// where a node has kHubDegree incidences or more on average (the updates' atomics then meet on few
// nodes).  5M x 5M row-net, us of updates a level at P / 8, P / 32, P / 128: 1370 incidences a node 1779,
// 2010, 2475; 2460 a node 2398, 1988, 2023; 4100 a node 2779, 2002, 1274; 5800 a node 3275, 1567, 1063.
constexpr int kMoveFull = 8, kMoveFullHubs = 128, kHubDegree = 2048;
// On levels of at most kLoopSoloNodes nodes the cluster launch recounts above P / kMoveCount moved incidences: the
// updates' atomics meet on the same gains, and no hyperedge is too wide for the warp that counts it (161 nodes, 110K
// pins: 39 us for the moves of a refinement selection; 150K-node netlist whose high-fanout nets are cut throughout 1.69
// ms a bisection, then 1.49; row-net of 30K nodes 1.83 and 1.71; at P / 16 1.5 % slower, at P / 4 the same).
constexpr int kMoveCount = 8;

// Refinement selections run on the whole grid on levels of more than kGridSelLarge nodes, and of more than
// kGridSelNodes nodes and kLoopAlonePins pins where the coarser level has kGridSelRatio times fewer nodes (its sides
// are a rough start, so many nodes move); the others stay in the cluster launch, whose steps are cheaper when few do.
// Bisections, cluster and grid: 5M-node row-net 55.8 and 53.6 ms; 155K-node netlist merged by its largest nets (HDH,
// four iterations) 1069 and 906 us, 600K-node row-net alike 2910 and 2658; 1M-node netlist 2753 and 2797, kept
// 500K-node hierarchy refined 2314 and 2521.
constexpr int kGridSelNodes = 1 << 17, kGridSelLarge = 1 << 21, kGridSelRatio = 8;

// What one selection leaves for the update after it; two are used in turn.
struct LoopRound {
    unsigned ents, items, cands, pad;
    unsigned long long inc;     // incidences of the moved nodes
    unsigned long long weight;  // node weight moved to side 1 less that moved to side 0
    unsigned ties[kLoopMaxCluster][2];
};

// Lives in the handle's small scratch.  The histogram and the rounds are zero at the start of a level
// (k_level_start, start_level); the side weights carry over from the coarser level.
struct LoopState {
    unsigned hist[2][kHistBins];
    LoopRound rd[2];
    unsigned cmd;      // next step of the helper blocks: 0 leave, else 1 | own << 1
    unsigned pending;  // the launch stopped after a selection too large for one cluster
    unsigned sel;      // which LoopRound the last selection used
    unsigned it;       // refinement iterations done
    unsigned status0;  // the level's rebalance ran out of candidates (the last level written is 0)
    unsigned long long W[2];  // side weights
    // a refinement selection by the grid (k_sel_count): whether it takes place, its groups' threshold gains
    // (mode 1: all, 2: from thr up), and how many of the ties at them when not all
    unsigned go, ticket, mode[2], thr[2], take[2];
    // a stop inside the rebalance: its state
    unsigned rebal, rounds;
    int heavy;
    long long room, need;
};

// A level's arrays as the gain update reads them.
struct MoveArgs {
    int N, E, P;
    const int *noff, *nadj, *hoff, *pins, *hw, *nw;
    uint8_t *side, *prev;
    int *gain;
    unsigned long long *pair;  // per hyperedge: pins on side 0 << 32 | pins on side 1
    LoopState *ls;
    int4 *ent;  // move list: node and its side now, incidences [y, z) (move_entry)
    int4 *items;
    int item_cap;
    int lanes;           // lanes per entry of the move list (8 or 32)
    int run, run_shift;  // incidences per entry (a power of two) and its logarithm
};

struct LoopParams {
    long long W, limit0, limit1, sq;
    int m0, m, iters;
    bool initial;  // Algorithm 3 first (all nodes on side 1)
    bool resume;   // continue after the grid took a pending update
    bool pending;  // resume: the grid's last selection (if it took place) is not in the gains yet
    bool suspend;  // large moves may be left to the grid
    bool start;    // the launch also projects the sides (from `coarse` by `cmap`) and counts the gains
    const int *cmap;
    const uint8_t *coarse;
};
void launch_refine_loop(cudaStream_t s, const MoveArgs &m, const LoopParams &p, unsigned long long *cand,
                        uint32_t *status,
                        unsigned *pending_slot);

}  // namespace bp
