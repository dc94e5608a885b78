"""The one-block refinement's split of a level's hyperedges: a thread up to 8 pins, eight lanes up to 32, a warp above,
with the pins in shared memory and without.  Degrees at the edges, each kind alone and all together, counts around
the four hyperedges a warp takes at once, weights.  Integer arithmetic: identical to the oracle's."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _csr(N, degs, seed, hw_max=1, nw_max=1):
    rng = np.random.default_rng(seed)
    hoff = np.zeros(len(degs) + 1, np.int32)
    hoff[1:] = np.cumsum(degs)
    pins = np.concatenate([rng.choice(N, size=d, replace=False) for d in degs]).astype(np.int32)
    return dict(N=N, E=len(degs), hoff=hoff, pins=pins,
                nw=rng.integers(1, nw_max + 1, size=N).astype(np.int32) if nw_max > 1 else None,
                hw=rng.integers(1, hw_max + 1, size=len(degs)).astype(np.int32) if hw_max > 1 else None)


EDGES = [7, 8, 9, 15, 16, 17, 24, 25, 31, 32, 33, 34, 63, 64, 65, 128, 129]
CASES = {
    "threads": (500, [8] * 700, 0.02),
    **{"groups_%d" % n: (400, [9] * n + [32] * n, 0.03) for n in (1, 3, 4, 5, 63, 64, 65)},
    "warps": (900, [33, 64, 300, 900] * 9, 0.02),
    "all": (1500, EDGES * 15 + [2, 3, 5] * 450, 0.01),
    # 12,000 nodes leave no room for the pins beside them
    "unstaged": (12_000, EDGES * 16 + [2] * 1500, 0.01),
}


@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("weighted", [False, True])
def test_hyperedge_split_matches_oracle(name, weighted):
    import paper_2012_13618_gb300 as bp
    n, degs, eps = CASES[name]
    assert sum(degs) <= 17_000
    g = _csr(n, degs, len(degs), 5 if weighted else 1, 3 if weighted else 1)
    ref = oracle.bisect(oracle.Hypergraph.from_dict(g), eps, "LDH", 6, 3)
    with bp.create_from(g) as h:
        for run in range(2):
            parts, st = h.partition(2, eps, "LDH", 6, 3)
            assert st == ref["status"] and np.array_equal(parts, ref["side"]), run
