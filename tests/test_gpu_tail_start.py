"""Where the coarse tail starts: at 25,000 pins, at 17,000 where the input has a hyperedge of more than 256 pins (before
duplicates are dropped).  A hypergraph the tail takes whole needs few launches.  Reloading a workspace and the children
of a k-way partition follow their own input.  Integer arithmetic: identical to the oracle's."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _csr(N, degs, seed):
    rng = np.random.default_rng(seed)
    hoff = np.zeros(len(degs) + 1, np.int32)
    hoff[1:] = np.cumsum(degs)
    pins = np.concatenate([rng.choice(N, size=d, replace=False) for d in degs]).astype(np.int32)
    return dict(N=N, E=len(degs), hoff=hoff, pins=pins, nw=None, hw=None)


@pytest.mark.parametrize("wide,rest,whole", [(256, 6180, True), (257, 6180, False), (257, 4180, True), (256, 6300, False)])
def test_start_follows_the_widest_hyperedge(wide, rest, whole):
    import paper_2012_13618_gb300 as bp
    g = _csr(3000, [wide] + [4] * (rest - 1), rest)
    ref = oracle.bisect(oracle.Hypergraph.from_dict(g), 0.03, "LDH", 25, 2)
    with bp.create_from(g) as h:
        n = bp.kernel_launches()
        for run in range(3):
            parts, st = h.partition(2, 0.03, "LDH", 25, 2)
            assert st == ref["status"] and np.array_equal(parts, ref["side"]), run
            if run == 0:
                assert (bp.kernel_launches() - n < 8) == whole
    # a 4-way partition and a server's worker that takes both kinds in turn
    other = _csr(3000, [4] * 6000, 1)
    with bp.Server(workers=1) as srv:
        for x in (g, other, g):
            ref4, rst = oracle.partition(oracle.Hypergraph.from_dict(x), 4, 0.05, "LDH", 25, 2)
            got, st, _, _ = srv.wait(srv.submit(x, k=4, eps=0.05, policy="LDH", levels=25, iters=2))
            assert st == rst and np.array_equal(got, ref4)
