"""The cases of the cluster launch's work split with the coarse tail off, so that small levels reach the launch too: its
first block alone up to 4,096 nodes and all blocks above, Algorithm 3 on either, levels of no or one hyperedge,
thresholds beyond the histogram; and selections of more nodes of long incidence lists than one pass of a flush holds.
Integer arithmetic: the partition and the status must be identical to the oracle's."""
import os
import subprocess
import sys

import pytest

import synth

pytestmark = pytest.mark.gpu

_ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _cases():
    from test_gpu_refine_loop import CASES, _csr
    yield from CASES.items()
    for n in (4095, 4096, 4097, 4128):
        for levels in (0, 1, 25):
            yield "split_%d_%d" % (n, levels), (lambda n=n: synth.uniform(n, n + 100, 2, 6, seed=n), 0.02, levels, 3)
    # 600 nodes of 670 incidences each, half of which move in one selection
    yield "hubs", (lambda: _csr(600, [2] * 200_000, 12, nw_max=2), 0.02, 0, 3)
    yield "hubs_shared", (lambda: _csr(5000, [9] * 300_000, 13), 0.02, 0, 2)


_CHILD = """
import sys
sys.path[:0] = [%r, %r]
import numpy as np
import oracle
import paper_2012_13618_gb300 as bp
from test_gpu_refine_loop_grid import _cases
n = 0
for name, (gen, eps, levels, iters) in _cases():
    g = gen()
    ref = oracle.bisect(oracle.Hypergraph.from_dict(g), eps, "LDH", levels, iters)
    with bp.create_from(g) as h:
        for run in range(3):
            parts, st = h.partition(2, eps, "LDH", levels, iters)
            assert st == ref["status"] and np.array_equal(parts, ref["side"]), (name, run)
        assert h.plan_active(), name
        parts, st = h.refine_kept(eps, iters)
        assert st == ref["status"] and np.array_equal(parts, ref["side"]), name
    n += 1
print("same", n)
"""


def test_work_split_without_the_tail():
    r = subprocess.run([sys.executable, "-c", _CHILD % (_ROOT, os.path.join(_ROOT, "tests"))], cwd=_ROOT,
                       env={**os.environ, "BIPART_TAIL_NODES": "0"}, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
    assert "same %d" % len(list(_cases())) in r.stdout
