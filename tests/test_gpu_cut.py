"""bipart_cut_noalloc at the degrees where a hyperedge goes from one thread to a warp to a block, against the
oracle's cut (integers: equal)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 2, 33, 64])
@pytest.mark.parametrize("copies", [1, 400])
def test_cut_noalloc_degree_edges(k, copies):
    import torch
    import paper_2012_13618_gb300 as bp
    rng = np.random.default_rng(100 * k + copies)
    N = 20_011
    degs = [0, 1, 2, 3, 4, 5, 31, 32, 33, 64, 511, 512, 513, 4097, 9001] * copies
    hoff = np.zeros(len(degs) + 1, np.int32)
    hoff[1:] = np.cumsum(degs)
    pins = rng.integers(0, N, size=int(hoff[-1])).astype(np.int32)  # repeated pins among them
    hw = rng.integers(1, 6, size=len(degs)).astype(np.int32)
    parts = (np.arange(N) * k // N).astype(np.int32)
    ref = oracle.cut(oracle.Hypergraph.from_csr(N, hoff, pins, None, hw), parts)
    d = [torch.from_numpy(x).cuda() for x in (hoff, pins, hw, parts)]
    out = torch.full((1,), -7, dtype=torch.int64, device="cuda")
    for _ in range(2):
        bp.cut_noalloc(N, d[0], d[1], d[2], d[3], k, out)
        assert int(out.item()) == ref
    bad = parts.copy()
    bad[pins[hoff[-2]]] = k  # a part out of range, met by the widest hyperedge
    bp.cut_noalloc(N, d[0], d[1], d[2], torch.from_numpy(bad).cuda(), k, out)
    assert int(out.item()) == -1
