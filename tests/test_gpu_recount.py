"""Moves of a large share of a level's incidences: the cluster launch counts the gains afresh instead of updating them.
Levels of few nodes and many pins up to the 4,096 nodes of one selecting block, and levels above, which go on
updating; gains that add up in shared memory and gains that do not, wide and narrow hyperedges, weights.  Grid path alone (the coarse tail off) beside the
default.  Integer arithmetic: identical to the oracle's."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

_ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _csr(N, degs, seed, hw_max=1, nw_max=1):
    rng = np.random.default_rng(seed)
    hoff = np.zeros(len(degs) + 1, np.int32)
    hoff[1:] = np.cumsum(degs)
    pins = np.concatenate([rng.choice(N, size=d, replace=False) for d in degs]).astype(np.int32)
    return dict(N=N, E=len(degs), hoff=hoff, pins=pins,
                nw=rng.integers(1, nw_max + 1, size=N).astype(np.int32) if nw_max > 1 else None,
                hw=rng.integers(1, hw_max + 1, size=len(degs)).astype(np.int32) if hw_max > 1 else None)


def _cases():
    # few nodes, thousands of incidences each: one selecting block, gains summed in shared memory
    yield "few", _csr(60, [2, 3] * 6000, 1), 0.02, 2, 3
    yield "few_weighted", _csr(160, [2, 3, 5] * 8000, 2, hw_max=7, nw_max=6), 0.01, 2, 3
    yield "wide", _csr(400, [2] * 9000 + [31, 32, 33, 64, 400] * 40, 3, nw_max=3), 0.01, 3, 3
    # 8 and 9 incidences a node (added up globally, in shared memory), the largest such level and the next
    yield "sums_8", _csr(4096, [4] * 8192, 4, nw_max=3), 0.02, 0, 4
    yield "sums_9", _csr(4096, [4] * 9000, 5, nw_max=3), 0.02, 0, 4
    yield "above", _csr(4097, [4] * 9000, 8, nw_max=3), 0.02, 0, 4
    # more nodes than the shared-memory sums hold
    yield "many", _csr(20_000, [12] * 20_000, 6), 0.02, 1, 4
    # Algorithm 3 on a level of hubs
    yield "initial", _csr(90, [3] * 10_000, 7), 0.02, 0, 2


_CHILD = """
import sys
sys.path[:0] = [%r, %r]
import numpy as np
import oracle
import paper_2012_13618_gb300 as bp
from test_gpu_recount import _cases
n = 0
for name, g, eps, levels, iters in _cases():
    ref = oracle.bisect(oracle.Hypergraph.from_dict(g), eps, "LDH", levels, iters)
    with bp.create_from(g) as h:
        for run in range(3):
            parts, st = h.partition(2, eps, "LDH", levels, iters)
            assert st == ref["status"] and np.array_equal(parts, ref["side"]), (name, run)
    n += 1
print("same", n)
"""


@pytest.mark.parametrize("env", [{}, {"BIPART_TAIL_NODES": "0"}], ids=["default", "grid_alone"])
def test_recounted_gains_match_oracle(env):
    r = subprocess.run([sys.executable, "-c", _CHILD % (_ROOT, os.path.join(_ROOT, "tests"))], cwd=_ROOT,
                       env={**os.environ, **env}, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
    assert "same %d" % len(list(_cases())) in r.stdout
