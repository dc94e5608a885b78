"""Levels of many nodes and few pins: started by the grid above 65,536 nodes whatever their pins, refined by it above
2,097,152, and with no pins at all on the coarsest level.  As a coarsest level of more nodes than the tie bitmaps of
the cluster hold, Algorithm 3 and the refinement rank their ties window by window.  A node heavier than all others
keeps Algorithm 3 to a few rounds.  Integer arithmetic: identical to the oracle's."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _sparse(N, E, seed, heavy=True):
    rng = np.random.default_rng(seed)
    nw = np.ones(N, np.int32)
    if heavy:
        nw[rng.integers(0, 1000)] = N + 7
    return dict(N=N, E=E, hoff=np.arange(0, 2 * E + 1, 2, dtype=np.int32),
                pins=rng.choice(N, size=2 * E, replace=False).astype(np.int32), nw=nw, hw=None)


def _paired():
    # the first 131,100 nodes in pairs: the others' gains are higher, so the first block's ties lie in its second window
    N = 2_100_001
    nw = np.ones(N, np.int32)
    nw[131_150] = N + 7
    return dict(N=N, E=65_550, hoff=np.arange(0, 131_101, 2, dtype=np.int32), pins=np.arange(131_100, dtype=np.int32),
                nw=nw, hw=None)


CASES = {
    "start_65536": (lambda: _sparse(65_536, 3000, 1, heavy=False), 3, 2),
    "start_65537": (lambda: _sparse(65_537, 3000, 2, heavy=False), 3, 2),
    "no_pins": (lambda: _sparse(70_001, 1, 3, heavy=False), 3, 1),
    "no_hyperedges": (lambda: _sparse(70_001, 0, 4, heavy=False), 3, 1),
    "grid_selects": (lambda: _sparse(2_100_001, 9000, 5), 1, 2),
    "windows": (_paired, 0, 2),
}


@pytest.mark.parametrize("name", CASES)
def test_many_nodes_few_pins_match_oracle(name):
    import paper_2012_13618_gb300 as bp
    gen, levels, iters = CASES[name]
    g = gen()
    ref = oracle.bisect(oracle.Hypergraph.from_dict(g), 0.05, "LDH", levels, iters)
    with bp.create_from(g) as h:
        for run in range(3):
            parts, st = h.partition(2, 0.05, "LDH", levels, iters)
            assert st == ref["status"] and np.array_equal(parts, ref["side"]), run
        assert h.plan_active()
