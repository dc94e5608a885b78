"""Long stretches of nodes that are in no hyperedge (and levels that are nearly all of them) through the
load-balanced passes, which step over empty segments in doubling steps.  Integer arithmetic: the partition and the
status must be identical to the oracle's."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _at(N, nodes, E, d, seed):
    """E hyperedges of d distinct pins among `nodes`; the other nodes are in none."""
    rng = np.random.default_rng(seed)
    nodes = np.asarray(nodes, np.int32)
    pins = np.concatenate([nodes[np.sort(rng.choice(nodes.size, d, replace=False))] for _ in range(E)])
    return dict(N=N, E=E, hoff=(np.arange(E + 1) * d).astype(np.int32), pins=pins.astype(np.int32), nw=None, hw=None)


CASES = {
    "ends": lambda: _at(50_000, [0, 1, 49_998, 49_999], 40, 3, 1),
    "powers": lambda: _at(70_000, [2 ** k + q for k in range(17) for q in (-1, 0, 1) if 2 ** k + q < 70_000], 3000, 4, 2),
    "every_1000th": lambda: _at(400_000, range(7, 400_000, 1000), 40_000, 5, 3),
    "two_clumps": lambda: _at(150_000, list(range(300)) + list(range(149_000, 149_300)), 60_000, 3, 4),
}


@pytest.mark.parametrize("policy", ["LDH", "RAND"])
@pytest.mark.parametrize("name", CASES)
def test_gaps_match_oracle(name, policy):
    import paper_2012_13618_gb300 as bp
    g = CASES[name]()
    ref = oracle.bisect(oracle.Hypergraph.from_dict(g), 0.05, policy, 6, 2)
    with bp.create_from(g) as h:
        for run in range(3):
            parts, st = h.partition(2, 0.05, policy, 6, 2)
            assert st == ref["status"] and np.array_equal(parts, ref["side"]), run
