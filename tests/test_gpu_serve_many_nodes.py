"""A request of many nodes and few hyperedges stays within the server's admission estimate: the refinement's lists and
gains live in the coarsening's scratch."""
import numpy as np
import pytest

from test_gpu_serve_budget import counting, estimate_bytes  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hedges", [1, 1000])
def test_many_nodes_within_the_estimate(counting, hedges):  # noqa: F811
    import paper_2012_13618_gb300 as bp
    N = 1_000_003
    rng = np.random.default_rng(4)
    g = dict(N=N, E=hedges, hoff=np.arange(0, 2 * hedges + 1, 2, dtype=np.int32),
             pins=rng.choice(N, size=2 * hedges, replace=False).astype(np.int32), nw=None, hw=None)
    live = counting.live
    counting.reset_peak()
    with bp.Server(workers=1) as srv:
        got, st, _, _ = srv.wait(srv.submit(g, k=2, eps=0.05, policy="LDH", levels=1, iters=2))
    ones = int(got.sum())
    assert st == 0 and max(ones, N - ones) <= int(N * 1.05 / 2)
    assert counting.peak - live <= estimate_bytes(g)
