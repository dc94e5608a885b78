"""The gain update's and the rebalance's edges: move-list runs of 16 and 64 incidences, hyperedges walked by a
warp or queued, whole recounts on levels of few nodes with many incidences, and rebalance rounds that start from
the last threshold on levels wide enough for the grouped scan (more than 4,096 nodes a block).  Integer
arithmetic: the partition and the status must be identical to the oracle's."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _csr(N, degs, seed, nw=None, skew=0, hw_max=1):
    rng = np.random.default_rng(seed)
    hoff = np.zeros(len(degs) + 1, np.int32)
    hoff[1:] = np.cumsum(degs)
    pins = []
    for d in degs:
        p = rng.choice(N, size=d, replace=False)
        if skew and d < skew:  # hub nodes: one pin among the first `skew` nodes
            p[0] = rng.integers(0, skew)
            p = np.unique(p)
            while len(p) < d:
                p = np.unique(np.append(p, rng.integers(0, N)))
        pins.append(p)
    pins = np.concatenate(pins).astype(np.int32)
    return dict(N=N, E=len(degs), hoff=hoff, pins=pins, nw=nw,
                hw=rng.integers(1, hw_max + 1, size=len(degs)).astype(np.int32) if hw_max > 1 else None)


def _heavy_tail(n, seed):
    rng = np.random.default_rng(seed)
    w = np.ones(n, np.int32)
    w[rng.integers(0, n, n // 50)] = 400
    return w


CASES = {
    # P <= 16 N: runs of 16; hub nodes of several runs; hyperedges around the walk's and the queue's limits
    "short_runs": (lambda: _csr(9000, [2, 3, 15, 16, 17] * 1600 + [63, 64, 65, 128, 511, 512, 513] * 3, 1, skew=50), 0.005, 25, 3),
    # P > 16 N: runs of 64
    "long_runs": (lambda: _csr(2000, [5, 20, 33] * 2000 + [64, 65, 512, 513] * 4, 2, skew=20, hw_max=5), 0.005, 25, 3),
    # more than 2,048 incidences a node and more pins than the cluster updates alone
    "hubs": (lambda: _csr(150, [4] * 90_000, 3), 0.01, 0, 3),
    # grouped scans: the imbalance of hub columns takes many rounds; node weights above and below the room
    "scan_rownet": (lambda: synth.rownet(150_000, 150_000, seed=5), 0.001, 4, 2),
    "scan_weighted": (lambda: dict(synth.rownet(140_001, 140_001, seed=6), nw=_heavy_tail(140_001, 7)), 0.0001, 3, 2),
    "scan_uniform": (lambda: synth.uniform(200_003, 150_000, 2, 6, seed=8), 0.0, 2, 3),
}


@pytest.mark.parametrize("name", CASES)
def test_moves_match_oracle(name):
    import paper_2012_13618_gb300 as bp
    gen, eps, levels, iters = CASES[name]
    g = gen()
    ref = oracle.bisect(oracle.Hypergraph.from_dict(g), eps, "LDH", levels, iters)
    with bp.create_from(g) as h:
        for run in range(3):
            parts, st = h.partition(2, eps, "LDH", levels, iters)
            assert st == ref["status"] and np.array_equal(parts, ref["side"]), run
