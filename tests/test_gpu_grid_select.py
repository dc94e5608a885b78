"""Refinement selections by the whole grid (levels of more than 131,072 nodes over one an eighth as large, or of more
than 2,097,152): just above the limits and below them, ties spread over all blocks, thresholds in the histogram's clamped ends (left to the cluster
launch, at the first iteration or a later one), hub nodes, node weights, several iterations.  Integer
arithmetic: the partition and the status must be identical to the oracle's."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _netlist(N, seed, hw_max=1, heavy=0, unit=False):
    """Merged by its largest nets (HDH) into a level far smaller: the grid's selections."""
    g = synth.netlist(N, int(1.2 * N), seed, wmax=1 if unit else 4)
    rng = np.random.default_rng(seed)
    if hw_max > 1:
        g["hw"] = rng.integers(1, hw_max + 1, size=g["E"]).astype(np.int32)
    if heavy:  # a few hyperedges whose gains leave the histogram
        g["hw"] = np.ones(g["E"], np.int32)
        g["hw"][rng.integers(0, g["E"], heavy)] = 5000
    return g


CASES = {
    "at_limit": (lambda: _netlist(131_072, 1), "HDH", 0.05, 2, 2),
    "above_limit": (lambda: _netlist(131_073, 2), "HDH", 0.05, 2, 5),
    "ties": (lambda: _netlist(300_007, 3, unit=True), "HDH", 0.03, 2, 3),
    "clamped": (lambda: _netlist(140_000, 4, hw_max=10_000), "HDH", 0.05, 2, 2),
    "some_clamped": (lambda: _netlist(140_000, 5, heavy=2000), "HDH", 0.05, 2, 4),
    "hubs": (lambda: synth.rownet(300_000, 300_000, seed=6), "HDH", 0.1, 3, 4),
    "large": (lambda: synth.uniform(2_100_000, 1_200_000, 2, 4, seed=8), "LDH", 0.1, 20, 1),
    "slowly_merged": (lambda: synth.uniform(300_007, 280_000, 2, 2, seed=3), "RAND", 0.03, 2, 3),
    "no_iterations": (lambda: _netlist(140_000, 7), "HDH", 0.05, 2, 0),
}


@pytest.mark.parametrize("name", CASES)
def test_grid_selection_matches_oracle(name):
    import paper_2012_13618_gb300 as bp
    gen, policy, eps, levels, iters = CASES[name]
    g = gen()
    ref = oracle.bisect(oracle.Hypergraph.from_dict(g), eps, policy, levels, iters)
    with bp.create_from(g) as h:
        for run in range(3):
            parts, st = h.partition(2, eps, policy, levels, iters)
            assert st == ref["status"] and np.array_equal(parts, ref["side"]), run
        parts, st = h.refine_kept(eps, iters)
        assert st == ref["status"] and np.array_equal(parts, ref["side"])
