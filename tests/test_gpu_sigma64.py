"""FP64 sigma vector (element by element from the string links) against the
oracle, on vectors without alpha-beta symmetry, at the sizes where its plan
changes: one string, no links, one and several chunks of a row's links, odd
link counts, different alpha and beta strings.

sigma_I sums at most n_off^2 + 2 n_off + 2 nnz terms (below 4,000 here) of
magnitude |g'| |c|, so FP64 rounding stays below 4000 * 2^-53 of the largest
element times a modest cancellation factor: 1e-11 of the largest element.
"""
import numpy as np
import pytest

import mbe_synth as ms
from oracle import casci as oc

from test_gpu_open_shell import core_signs as core_signs_ab

pytestmark = pytest.mark.gpu
TOL = 1e-11


@pytest.fixture(scope="module")
def lib():
    from paper_1905_02786_gb300 import build, _binding
    build.build()
    _binding.load_library()
    return _binding


@pytest.mark.parametrize("norb,na,nb,act", [
    (3, 1, 1, [0]),                                  # one determinant, no links
    (5, 3, 0, [0, 1, 2, 3]),                         # no beta electron
    (6, 3, 3, [0, 1, 2]),                            # all strings full
    (13, 1, 1, list(range(13))),                     # 13 strings, 12 links
    (8, 3, 3, list(range(8))),                       # 15 links (odd)
    (12, 5, 3, list(range(12))),                     # 792 x 220 strings
    (12, 5, 5, list(range(12))),                     # two chunks of 18 and 17 links
    (13, 5, 5, list(range(13))),                     # three chunks
    (14, 6, 6, list(range(14))),                     # eight chunks, 3,003 strings
])
def test_sigma64_rows_vs_oracle(lib, norb, na, nb, act):
    h, eri, _ = ms.gen_integrals(norb, na, 41)
    nocc = na if na == nb else (na, nb)
    sp = oc.Space(h, eri, nocc, act)
    rng = np.random.default_rng(5)
    c = rng.standard_normal(sp.ndet)
    m = lib.MBE(0, spin_shift=0.5)
    m.load(h, eri, na + nb, two_sz=na - nb)
    sig, ecore = lib.mbe_sigma(m.ctx, act, c)
    m.close()
    S = core_signs_ab(sp, nb, act)
    cs = S * c
    rows = np.unique(np.concatenate([rng.integers(0, sp.ndet, 600), [0, sp.ndet - 1]]))
    ref = S[rows] * (sp.sigma_rows(cs, rows) + 0.5 * sp.s2(cs)[rows]) - ecore * c[rows]
    assert np.abs(sig[rows] - ref).max() <= TOL * np.abs(ref).max()
