"""The coarse tail takes hypergraphs of up to 35,000 pins and 6,144 nodes, or 25,000 pins and 12,288 nodes, whole, with the
pins in shared memory and without; one pin or node more is coarsened on the grid first.  Integer arithmetic: identical to the oracle's."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,pins,whole", [(3000, 35_000, True), (3000, 35_001, False), (6144, 35_000, True),
                                          (6145, 25_001, False), (6145, 25_000, True), (12_288, 25_000, True),
                                          (12_289, 24_999, False)])
def test_tail_limits_match_oracle(N, pins, whole):
    import paper_2012_13618_gb300 as bp
    rng = np.random.default_rng(pins + N)
    degs = [5] * (pins // 5 - 1)
    degs.append(pins - sum(degs))
    hoff = np.zeros(len(degs) + 1, np.int32)
    hoff[1:] = np.cumsum(degs)
    p = np.concatenate([rng.choice(N, size=d, replace=False) for d in degs]).astype(np.int32)
    g = dict(N=N, E=len(degs), hoff=hoff, pins=p, nw=rng.integers(1, 4, size=N).astype(np.int32), hw=None)
    ref = oracle.bisect(oracle.Hypergraph.from_dict(g), 0.02, "LDH", 25, 2)
    with bp.create_from(g) as h:
        n = bp.kernel_launches()
        for run in range(3):
            parts, st = h.partition(2, 0.02, "LDH", 25, 2)
            assert st == ref["status"] and np.array_equal(parts, ref["side"]), run
            if run == 0:
                assert (bp.kernel_launches() - n < 8) == whole
