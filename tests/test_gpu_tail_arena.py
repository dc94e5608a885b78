"""A hypergraph that coarsens slowly outgrows the coarse tail's first arena: the first call runs the tail again with a
larger one, and the second call still captures the plan.  Integer arithmetic: identical to the oracle's."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("levels", [25, 60])
def test_tail_arena_grows_and_the_second_call_captures(levels):
    import paper_2012_13618_gb300 as bp
    # a path whose edges weigh more from left to right: every node but the first takes its left edge, so a
    # contraction merges three nodes and leaves the others alone (25 levels of about 24,000 pins)
    n = 12_000
    g = dict(N=n, E=n - 1, hoff=np.arange(0, 2 * n - 1, 2, dtype=np.int32),
             pins=np.stack([np.arange(n - 1), np.arange(1, n)], 1).astype(np.int32).ravel(), nw=None,
             hw=np.arange(1, n, dtype=np.int32))
    ref = oracle.bisect(oracle.Hypergraph.from_dict(g), 0.05, "LWD", levels, 2)
    with bp.create_from(g) as h:
        for run in range(3):
            parts, st = h.partition(2, 0.05, "LWD", levels, 2)
            assert st == ref["status"] and np.array_equal(parts, ref["side"]), run
            assert h.plan_active() == (run > 0), run
        assert h.num_levels() == levels + 1
