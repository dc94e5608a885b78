"""Device memory from an allocator that hands out exact pieces off a 16-byte boundary, in workspaces reused at sizes
that just fit: a server's worker and the single child workspace of a one-lane k-way partition.  Integer
arithmetic: every result must be identical to the oracle's."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


class Offset:
    """Allocator hooks over PyTorch's caching allocator that shift every pointer by a few bytes."""

    def __init__(self, bp, shift):
        import torch
        self.torch, self.shift, self.live = torch, shift, {}
        self.a, self.f = bp._ALLOC(self._alloc), bp._FREE(self._free)

    def _alloc(self, ctx, nbytes, stream):
        try:
            p = int(self.torch.cuda.caching_allocator_alloc(int(nbytes) + self.shift, 0, int(stream or 0))) + self.shift
        except Exception:
            return None
        self.live[p] = int(nbytes)
        return p

    def _free(self, ctx, ptr, nbytes, stream):
        assert self.live.pop(int(ptr)) == int(nbytes)
        self.torch.cuda.caching_allocator_delete(int(ptr) - self.shift)


@pytest.mark.parametrize("shift", [4, 8])
def test_offset_allocator_matches_oracle(shift):
    import paper_2012_13618_gb300 as bp
    off = Offset(bp, shift)
    bp._check(bp.load().bipart_set_allocator(off.a, off.f, None))
    try:
        with bp.Server(workers=1) as srv:
            # 45,065 nodes fit what 40,001 left room for to the byte
            for n, k in ((40_001, 2), (45_065, 2), (6_001, 2), (45_065, 4), (6_003, 4)):
                g = synth.c3_instance(3, N=n)
                got, st, _, _ = srv.wait(srv.submit(g, k=k, eps=0.01, policy="LDH", levels=25, iters=2))
                ref, rst = oracle.partition(oracle.Hypergraph.from_dict(g), k, 0.01, "LDH", 25, 2)
                assert np.array_equal(got, ref) and st == rst, (n, k)
        g = synth.rownet(20_001, 20_001, seed=5)
        ref = oracle.bisect(oracle.Hypergraph.from_dict(g), 0.02, "LDH", 25, 2)
        with bp.create_from(g) as h:
            for run in range(3):
                parts, st = h.partition(2, 0.02, "LDH", 25, 2)
                assert st == ref["status"] and np.array_equal(parts, ref["side"]), run
            parts, st = h.refine_kept(0.02, 2)
            assert st == ref["status"] and np.array_equal(parts, ref["side"])
    finally:
        bp.load().bipart_batch_release()
        bp.use_default_allocator()
    assert not off.live
