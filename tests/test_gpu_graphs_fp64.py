"""CUDA-graph replay of the FP64 Davidson iteration and of the FP64 exact
points of the mixed one: the same kernels on the same data as plain launches,
hence the same bits, with and without restarts of a small subspace, closed and
open shell, and as the first call of a process (every one-time set-up then falls
into this call, before its first capture).
"""
import os
import subprocess
import sys

import numpy as np
import pytest

import mbe_synth as ms

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    from paper_1905_02786_gb300 import build, _binding
    build.build()
    _binding.load_library()
    return _binding


def _solve(lib, norb, nel, two_sz, ref, tuples, **opts):
    h, eri, _ = ms.gen_integrals(norb, (nel - two_sz) // 2, 53)
    m = lib.MBE(0, **opts)
    m.load(h, eri, nel, two_sz=two_sz)
    lib.mbe_set_reference(m.ctx, ref, [p for p in range(norb) if p not in ref])
    lib.mbe_reset_stats(m.ctx)
    tuples = np.array(tuples, dtype=np.int32)
    eps, st = lib.mbe_solve_tuples(m.ctx, tuples, tuples.shape[1])
    stats = lib.mbe_get_stats(m.ctx)
    m.close()
    assert np.all(st == 0)
    return eps, stats


@pytest.mark.parametrize("nel,two_sz", [(8, 0), (7, 1)])
@pytest.mark.parametrize("max_subspace", [4, 7, 20])
def test_same_bits(lib, nel, two_sz, max_subspace):
    tuples = [[6, 7], [6, 8], [7, 9], [0, 10]]
    run = [_solve(lib, 11, nel, two_sz, [1, 2, 3, 4, 5], tuples, graphs=g,
                  max_subspace=max_subspace) for g in (0, 1)]
    assert np.array_equal(run[0][0], run[1][0])
    a, b = run[0][1], run[1][1]
    assert a["iters_total"] == b["iters_total"] and a["launches"] == b["launches"]
    assert a["iters_max"] > max_subspace or max_subspace == 20    # it restarted
    assert a["graph_launches"] == 0 and b["graph_launches"] > 0
    assert b["host_launches"] < b["launches"] // 2


FIRST = """
import sys
sys.path[:0] = [{root!r}, {tests!r}]
from paper_1905_02786_gb300 import _binding as B
B.load_library()
from test_gpu_graphs_fp64 import _solve
print(*[float(x).hex() for x in _solve(B, 14, 6, 0, [0, 1, 2], [list(range(3, 13))], **{opts!r})[0]])
"""


@pytest.mark.parametrize("opts", [dict(precision=1), dict(precision=0), dict(precision=1, pspace=0)])
def test_first_call_of_a_process(lib, opts):
    """6e/13o: tensor-core sigma vectors with FP64 exact points in mixed mode."""
    code = FIRST.format(root=ROOT, tests=os.path.join(ROOT, "tests"), opts=opts)
    out = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr
    got = [float.fromhex(x) for x in out.stdout.split()]
    want, _ = _solve(lib, 14, 6, 0, [0, 1, 2], [list(range(3, 13))], graphs=0, **opts)
    assert np.array_equal(got, want)
