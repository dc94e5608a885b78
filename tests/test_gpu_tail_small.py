"""Small levels on both paths: refined by one block on shared memory (the cluster tail) and, with the tail
switched off, by the grid's refinement launch.  Sizes around the edges of the one-block pass: hyperedges of
one thread (up to 32 pins, in batches of four) and of a warp, counts around the block's width, levels whose
pins fit shared memory and levels whose pins do not, weights, gains beyond the clamped histogram.  Integer
arithmetic: the partition and the status must be identical to the oracle's."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

_ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _csr(N, degs, seed, hw_max=1, nw_max=1):
    rng = np.random.default_rng(seed)
    degs = [min(d, N) for d in degs]
    hoff = np.zeros(len(degs) + 1, np.int32)
    hoff[1:] = np.cumsum(degs)
    pins = np.concatenate([rng.choice(N, size=d, replace=False) for d in degs] or [np.zeros(0)]).astype(np.int32)
    return dict(N=N, E=len(degs), hoff=hoff, pins=pins,
                nw=rng.integers(1, nw_max + 1, size=N).astype(np.int32) if nw_max > 1 else None,
                hw=rng.integers(1, hw_max + 1, size=len(degs)).astype(np.int32) if hw_max > 1 else None)


def _cases():
    yield "one", _csr(1, [1], 1), 0.1, 3, 2
    yield "two", _csr(2, [2, 2, 1], 2, hw_max=3), 0.1, 3, 2
    yield "no_hyperedges", _csr(40, [], 3, nw_max=5), 0.05, 3, 2
    yield "batches", _csr(300, [1, 2, 3, 4, 5, 7, 8, 9, 31, 32, 33, 34] * 10, 4), 0.03, 25, 3
    for E in (511, 512, 513, 2047, 2048, 2049):  # threads of the block, hyperedges of one round
        yield "hyperedges_%d" % E, _csr(700, [2, 3, 4, 5] * (E // 4) + [3] * (E % 4), 5 + E, nw_max=3), 0.02, 25, 3
    yield "wide", _csr(2500, [32, 33, 64, 100, 1000, 2500, 2] * 5, 6, hw_max=4, nw_max=4), 0.02, 25, 3
    yield "most_nodes", _csr(12_288, [2, 2, 2, 3] * 2700, 7), 0.02, 2, 2   # 24,300 pins
    yield "above_tail", _csr(5000, [5] * 5001, 8, nw_max=2), 0.02, 25, 2        # 25,005 pins
    yield "exact", _csr(1500, [2, 3, 5] * 700, 9, hw_max=300_000, nw_max=3), 0.02, 25, 3
    yield "scarce", _csr(64, [3] * 100, 10, nw_max=40), 0.001, 4, 3


_CHILD = """
import sys
sys.path[:0] = [%r, %r]
import numpy as np
import oracle
import paper_2012_13618_gb300 as bp
from test_gpu_tail_small import _cases
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


@pytest.mark.parametrize("env", [{}, {"BIPART_TAIL_PINS": "400000"}, {"BIPART_TAIL_NODES": "0"}],
                         ids=["default", "tail_from_larger", "grid_alone"])
def test_small_levels_match_oracle(env):
    r = subprocess.run([sys.executable, "-c", _CHILD % (_ROOT, os.path.join(_ROOT, "tests"))], cwd=_ROOT,
                       env={**os.environ, **env}, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
    assert "same %d" % len(list(_cases())) in r.stdout
