"""Contraction and incidence at the edges of their paths on large levels: hyperedges sorted by a block instead of
swept by bitmap windows (ids spread over two windows and over more, sizes around the sort's limits and its
powers of two, repeated pins), block-private counters on levels wider than two blocks an SM, and tile starts by
search.  Integer arithmetic: the partition and the status must be identical to the oracle's."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _random(N, degs, seed, stretch=None):
    rng = np.random.default_rng(seed)
    degs = np.asarray(degs, np.int64)
    hoff = np.zeros(degs.size + 1, np.int64)
    np.cumsum(degs, out=hoff[1:])
    pins = rng.integers(0, N, hoff[-1]).astype(np.int32)  # repeated pins included
    if stretch:  # every hyperedge reaches both ends of the id range
        wide = degs > 256
        pins[hoff[:-1][wide]] = 0
        pins[hoff[:-1][wide] + 1] = N - 1
    return dict(N=N, E=int(degs.size), hoff=hoff.astype(np.int32), pins=pins, nw=None, hw=None)


_EDGES = [257, 511, 512, 513, 1023, 1025, 2048, 2049, 4095, 4096, 4097, 6144, 6145, 8191, 8192, 8193, 30_000]
CASES = {
    "two_windows": lambda: _random(400_000, _EDGES * 2 + [3] * 700_000, 1, True),
    "many_windows": lambda: _random(1_300_000, _EDGES * 3 + [3] * 700_000, 2, True),
    "wide_counters": lambda: _random(24_577, [4] * 1_650_000, 3),        # 268 incidences a node
    "widest_counters": lambda: _random(53_248, [5] * 2_800_000, 4),      # 52 K nodes, 263 a node
    "beyond_counters": lambda: _random(53_249, [5] * 2_800_000, 5),
    "tiles_by_search": lambda: _random(3000, [9] * 43_000, 6),           # 129 incidences a node
}


@pytest.mark.parametrize("name", CASES)
def test_contraction_matches_oracle(name):
    import paper_2012_13618_gb300 as bp
    g = CASES[name]()
    ref = oracle.bisect(oracle.Hypergraph.from_dict(g), 0.9, "LDH", 8, 1)
    with bp.create_from(g) as h:
        for run in range(2):
            parts, st = h.partition(2, 0.9, "LDH", 8, 1)
            assert st == ref["status"] and np.array_equal(parts, ref["side"]), run
