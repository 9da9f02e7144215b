"""Mixed-precision energies where the exact points change their sigma: the fused
tensor-core one up to 12 orbitals, the FP64 one from the string links beyond
(13 orbitals; 14 with few and with half the electrons of its strings, one
electron), against the FP64 mode.  Both end in an FP64-grade Rayleigh quotient
of a vector converged to a relative residual of 2e-7, whose square bounds the
energy error: 1e-8 Eh.
"""
import numpy as np
import pytest

import mbe_synth as ms

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_1905_02786_gb300 import build, _binding
    build.build()
    _binding.load_library()
    return _binding


@pytest.mark.parametrize("n,nsig", [(12, 2), (13, 1), (13, 3), (14, 2), (14, 4)])
@pytest.mark.parametrize("graphs", [0, 1])
def test_energies_vs_fp64(lib, n, nsig, graphs):
    h, eri, _ = ms.gen_integrals(n + 1, nsig, 29)
    ref = list(range(nsig))
    exp = list(range(nsig, n + 1))
    tk = np.array([exp[:n - nsig], exp[1:]])
    eps = []
    for prec in (0, lib.MBE_MIXED_BF16X3):
        m = lib.MBE(0, precision=prec, graphs=graphs, spin_shift=0.5)
        m.load(h, eri, 2 * nsig)
        lib.mbe_set_reference(m.ctx, ref, exp)
        e, st = lib.mbe_solve_tuples(m.ctx, tk, n - nsig)
        assert np.all(st == 0)
        eps.append(np.array(e))
        m.close()
    assert np.abs(eps[1] - eps[0]).max() < 1e-8
