"""Davidson iterations of CASCIs whose two lowest symmetric states lie close
together: the Ritz step has to give the lowest pair to FP64 accuracy, or the
corrections stop reducing the residual and the iteration count grows.

The reference is the same iteration (lowest-diagonal start vector, diagonal
preconditioner, no restart below 32 vectors) on the dense matrix with numpy's
FP64 eigensolver; rounding moves the iteration that first meets a tolerance by
one or two, not more.
"""
import numpy as np
import pytest

import mbe_synth as ms
from oracle import casci as oc

pytestmark = pytest.mark.gpu
NORB, NOCC, SHIFT = 7, 3, 0.5


@pytest.fixture(scope="module")
def lib():
    from paper_1905_02786_gb300 import build, _binding
    build.build()
    _binding.load_library()
    return _binding


def integrals(scale, x, core):
    """Couplings between different orbitals times `scale`, the lowest virtual
    lowered by x (the closed shells of HOMO and LUMO then nearly cross), every
    orbital by `core` (theta as deep as an all-electron active space's)."""
    h, eri, _ = ms.gen_integrals(NORB, NOCC, 2)
    s = np.array([1.0 if p == q else scale for p in range(NORB) for q in range(p + 1)])
    h = scale * h + (1.0 - scale) * np.diag(np.diag(h)) - core * np.eye(NORB)
    h[NOCC, NOCC] -= x
    return h, eri * s[:, None] * s[None, :]


def reference_iterations(h, eri, tol_r, tol_e):
    sp = oc.Space(h, eri, NOCC, list(range(NORB)))
    P = sp.sym_basis()
    H = P.T @ (sp.hdense() @ P + SHIFT * np.array([sp.s2(P[:, k]) for k in range(P.shape[1])]).T)
    gap = np.diff(np.linalg.eigvalsh(H)[:2])[0]
    hd = (P * P).T @ (sp.hdiag() + SHIFT * sp.s2diag())   # of the determinants
    old = None
    V = np.eye(len(H))[[np.argmin(hd)]]
    for it in range(1, 32):
        w, Y = np.linalg.eigh(V @ H @ V.T)
        x = Y[:, 0] @ V
        r = H @ x - w[0] * x
        if old is not None and abs(w[0] - old) < tol_e and np.linalg.norm(r) < tol_r:
            return it, gap
        old = w[0]
        d = w[0] - hd
        t = r / np.where(np.abs(d) < 1e-8, np.copysign(1e-8, d), d)
        for _ in range(2):
            t -= V.T @ (V @ t)
        V = np.vstack([V, t / np.linalg.norm(t)])
    raise AssertionError("no convergence below 32 vectors")


@pytest.mark.parametrize("scale,x,core", [(0.1, 1.42061, 3.0), (0.05, 1.40366, 3.0),
                                          (0.02, 1.39882, 3.0), (0.05, 1.40366, 12.0)])
@pytest.mark.parametrize("tol_r,tol_e", [(1e-8, 1e-12), (1e-11, 1e-13)])
def test_fp64_iterations(lib, scale, x, core, tol_r, tol_e):
    h, eri = integrals(scale, x, core)
    want, gap = reference_iterations(h, eri, tol_r, tol_e)
    assert gap < 4e-3
    m = lib.MBE(0, conv_tol_r=tol_r, conv_tol_e=tol_e, spin_shift=SHIFT, max_subspace=32)
    m.load(h, eri, 2 * NOCC)
    lib.mbe_set_reference(m.ctx, list(range(NOCC)), list(range(NOCC, NORB)))
    lib.mbe_reset_stats(m.ctx)
    eps, st = lib.mbe_solve_tuples(m.ctx, np.array([list(range(NOCC, NORB))], dtype=np.int32),
                                   NORB - NOCC)
    stats = lib.mbe_get_stats(m.ctx)
    m.close()
    assert st[0] == 0
    assert abs(eps[0] - oc.casci(h, eri, NOCC, list(range(NORB)))) < 1e-10
    assert stats["iters_max"] <= want + 2, (stats["iters_max"], want, gap)
