"""The symmetric branches of the FP64 sigma from the string links (upper triangle
computed; packed result in the FP64 Davidson, full result at the mixed mode's
exact points) beyond 12 orbitals against the oracle: CASCI energies of all
orbitals of one seeded system each.  8e/13o takes several chunks of a row's links.

Tolerances: 1e-10 Eh for the FP64 mode (residual 1e-8, error its square over the
gap), 1e-8 Eh for the mixed mode (relative residual 2e-7).  The two larger
energies are oracle.casci's (74 s and 14 minutes on 8 cores):
    h, eri, _ = mbe_synth.gen_integrals(n, nsig, 61)
    oracle.casci.casci(h, eri, nsig, list(range(n)))
"""
import numpy as np
import pytest

import mbe_synth as ms
from oracle import casci as oc

pytestmark = pytest.mark.gpu
STORED = {(13, 3): -10.884046037674054, (13, 4): -17.034811351750147}


@pytest.fixture(scope="module")
def lib():
    from paper_1905_02786_gb300 import build, _binding
    build.build()
    _binding.load_library()
    return _binding


@pytest.mark.parametrize("n,nsig", [(13, 2), (14, 2), (13, 3), (13, 4)])
def test_energy_vs_oracle(lib, n, nsig):
    h, eri, _ = ms.gen_integrals(n, nsig, 61)
    want = STORED.get((n, nsig))
    if want is None:
        want = oc.casci(h, eri, nsig, list(range(n)))
    for prec, tol in ((lib.MBE_FP64, 1e-10), (lib.MBE_MIXED_BF16X3, 1e-8)):
        m = lib.MBE(0, precision=prec)
        m.load(h, eri, 2 * nsig)
        lib.mbe_set_reference(m.ctx, list(range(nsig)), list(range(nsig, n)))
        eps, st = lib.mbe_solve_tuples(m.ctx, np.array([list(range(nsig, n))], dtype=np.int32),
                                       n - nsig)
        m.close()
        assert st[0] == 0 and abs(eps[0] - want) < tol, (eps[0], want)
