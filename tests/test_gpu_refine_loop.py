"""The cluster launch that refines a level (selections, moves, gains kept current under moves) against the
oracle at the sizes where its work split changes: the first block alone or all of them, gains counted inside
the launch or by the grid, moves large enough to be left to the grid, wide hyperedges, nodes of no hyperedge,
thresholds beyond the histogram.  Four calls on one handle: the first may use the cluster tail, the second
runs every level on the grid, the third captures, the fourth replays.  Integer arithmetic: the partition and
the status must be identical."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _csr(N, degs, seed, hw_max=1, nw_max=1):
    rng = np.random.default_rng(seed)
    hoff = np.zeros(len(degs) + 1, np.int32)
    hoff[1:] = np.cumsum(degs)
    pins = np.concatenate([rng.choice(N, size=d, replace=False) for d in degs] or [np.zeros(0)]).astype(np.int32)
    return dict(N=N, E=len(degs), hoff=hoff, pins=pins,
                nw=rng.integers(1, nw_max + 1, size=N).astype(np.int32) if nw_max > 1 else None,
                hw=rng.integers(1, hw_max + 1, size=len(degs)).astype(np.int32) if hw_max > 1 else None)


CASES = {
    # nodes of no hyperedge only, and one hyperedge among them
    "isolated": (lambda: _csr(700, [3], 1, nw_max=3), 0.02, 25, 2),
    # the largest level one block selects for, the first one all blocks share, Algorithm 3 on it
    "solo_4096": (lambda: synth.uniform(4096, 4096, 2, 6, seed=3), 0.02, 0, 3),
    "shared_4097": (lambda: synth.uniform(4097, 4200, 2, 6, seed=4), 0.02, 0, 3),
    "no_iterations": (lambda: synth.c3_instance(5, N=9000), 0.01, 25, 0),
    # gains counted by the launch up to 131,072 pins, by the grid above
    "pins_below": (lambda: _csr(20_000, [4] * 32_768, 6), 0.03, 1, 2),
    "pins_above": (lambda: _csr(20_000, [4] * 32_768 + [2], 6), 0.03, 1, 2),
    # hyperedges around a warp, a work item and several items wide, weighted nodes
    "wide": (lambda: _csr(9000, [32, 33, 512, 513, 1024, 1025, 5000, 9000] * 6 + [2] * 4000, 7, nw_max=4), 0.01, 25, 3),
    # gains beyond the clamped histogram: the exact radix passes, in one block and in all
    "exact_solo": (lambda: _csr(3000, [2, 3, 5] * 1500, 8, hw_max=200_000), 0.02, 25, 3),
    "exact_shared": (lambda: _csr(12_000, [2, 3, 5] * 5000, 9, hw_max=200_000, nw_max=4), 0.02, 2, 3),
    # hub columns: moves of more incidences than the cluster takes, stopping the launch for the grid
    "stops": (lambda: synth.rownet(120_000, 120_000, seed=11), 0.03, 25, 3),
}


@pytest.mark.parametrize("name", CASES)
def test_refine_loop_matches_oracle(name):
    import paper_2012_13618_gb300 as bp
    gen, eps, levels, iters = CASES[name]
    g = gen()
    ref = oracle.bisect(oracle.Hypergraph.from_dict(g), eps, "LDH", levels, iters)
    with bp.create_from(g) as h:
        for run in range(4):
            parts, st = h.partition(2, eps, "LDH", levels, iters)
            assert st == ref["status"] and np.array_equal(parts, ref["side"]), run
        assert h.plan_active()
        parts, st = h.refine_kept(eps, iters)
        assert st == ref["status"] and np.array_equal(parts, ref["side"])
