"""Mixed-precision sigma over (N-1)-electron strings at the sizes where its plan
changes (5 to 12 orbitals, odd and even, one electron to one hole, a single
string, pair counts below and around its 128-row tiles, row lengths that are no
multiple of 4) and on both sides of its range (4 and 13 orbitals), against the
FP64 sigma, which the oracle pins element by element.

Operands are split into two BF16 parts (relative error 2^-17 each) and the
lo x lo products (2^-18) are left out: 2.3e-5 of sum |g'| |c|, which exceeds the
largest element of sigma by less than 8 here: 2e-4 of the largest element.
"""
import itertools

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


@pytest.mark.parametrize("n,nsig", [
    (4, 2), (5, 1), (5, 2), (5, 5), (6, 3), (6, 5), (7, 1), (7, 4), (8, 4), (8, 8), (9, 2),
    (9, 8), (10, 5), (11, 5), (11, 10), (12, 1), (12, 2), (12, 6), (12, 11), (13, 3),
])
@pytest.mark.parametrize("shift", [0.0, 0.5])
def test_sigma_vs_fp64(lib, n, nsig, shift):
    h, eri, _ = ms.gen_integrals(n, nsig, 17)
    nstr = len(list(itertools.combinations(range(n), nsig)))
    c = ms.random_symmetric_ci(nstr, 5)[0]
    sig = []
    for prec in (0, lib.MBE_MIXED_BF16X3):
        m = lib.MBE(0, precision=prec, spin_shift=shift)
        m.load(h, eri, 2 * nsig)
        sig.append(lib.mbe_sigma(m.ctx, list(range(n)), c)[0].reshape(nstr, nstr))
        m.close()
    assert np.abs(sig[1] - sig[0]).max() <= 2e-4 * np.abs(sig[0]).max()
    assert np.array_equal(sig[1], sig[1].T)


@pytest.mark.parametrize("n,nocc,ref,order", [
    (13, 2, [0, 1], 5),       # 462 batch elements of 2e..4e/7o: several per CTA
    (12, 3, [0, 1, 2], 6),    # 84 of 6e/9o: about one per CTA
    (12, 4, [0, 1, 2, 3], 6),  # 28 of 8e/10o: several CTAs per element
])
def test_batches_vs_fp64(lib, n, nocc, ref, order):
    h, eri, _ = ms.gen_integrals(n, nocc, 23)
    exp = [p for p in range(n) if p not in ref]
    tk = np.array(list(itertools.combinations(exp, order)))
    eps = []
    for prec in (0, lib.MBE_MIXED_BF16X3):
        m = lib.MBE(0, precision=prec)
        m.load(h, eri, 2 * nocc)
        lib.mbe_set_reference(m.ctx, ref, exp)
        e, st = lib.mbe_solve_tuples(m.ctx, tk, order)
        assert np.all(st == 0)
        eps.append(np.array(e))
        m.close()
    assert np.abs(eps[1] - eps[0]).max() < 1e-8
