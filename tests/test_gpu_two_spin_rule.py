"""Mixed-precision solves on both sides of the rule that chooses the kernel of
the two-spin part (rows of c, or pairs of (N-1)-electron strings): strings less
and more than half full, one tuple and a batch, against the FP64 mode.  Both end
in an FP64-grade Rayleigh quotient of a vector converged to a relative residual
of 2e-7, whose square bounds the energy error: 1e-8 Eh.
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


@pytest.mark.parametrize("norb,n,nsig,count", [
    (12, 5, 2, 91), (12, 5, 2, 92),        # 6 tiles of the rows of c per SM: one, then the other
    (12, 7, 2, 43), (12, 7, 2, 44),
    (14, 9, 4, 14), (14, 9, 4, 15),        # 12 per SM
    (13, 10, 5, 14), (14, 10, 5, 15),      # 48 per SM
    (12, 9, 5, 20),                        # twice as many tiles: rows of c
    (13, 11, 8, 8), (14, 12, 9, 8),        # more than half full: rows of c
    (12, 12, 5, 1), (12, 12, 7, 1), (14, 12, 7, 2),   # pull lists in global memory
])
def test_energies_vs_fp64(lib, norb, n, nsig, count):
    h, eri, _ = ms.gen_integrals(norb, nsig, 47)
    ref = list(range(nsig))
    tk = np.array(list(itertools.islice(itertools.combinations(range(nsig, norb), n - nsig), count)))
    eps = []
    for prec in (lib.MBE_FP64, lib.MBE_MIXED_BF16X3):
        m = lib.MBE(0, precision=prec)
        m.load(h, eri, 2 * nsig)
        lib.mbe_set_reference(m.ctx, ref, [p for p in range(norb) if p not in ref])
        e, st = lib.mbe_solve_tuples(m.ctx, tk, n - nsig)
        assert np.all(st == 0)
        eps.append(np.array(e))
        m.close()
    assert np.abs(eps[1] - eps[0]).max() < 1e-8


def test_bin_beyond_one_batch(lib):
    """4,845 tuples of 4e/6o with max_batch above that: the (N-1)-electron kernel
    takes 4,096 at a time, so the bin is solved as the two parts are, bit for bit."""
    norb, nsig, n = 22, 2, 6
    h, eri, _ = ms.gen_integrals(norb, nsig, 47)
    tk = np.array(list(itertools.combinations(range(2, norb), n - nsig)), dtype=np.int32)
    assert len(tk) == 4845

    def solve(part):
        m = lib.MBE(0, precision=lib.MBE_MIXED_BF16X3, max_batch=8192)
        m.load(h, eri, 2 * nsig)
        lib.mbe_set_reference(m.ctx, [0, 1], list(range(2, norb)))
        e, st = lib.mbe_solve_tuples(m.ctx, part, n - nsig)
        m.close()
        assert np.all(st == 0)
        return e

    assert np.array_equal(solve(tk), np.concatenate([solve(tk[:4096]), solve(tk[4096:])]))


@pytest.mark.parametrize("n,nsig", [(10, 4), (9, 6)])
def test_batch_and_alone(lib, n, nsig):
    """A tuple in a batch and alone: repeated calls give the same bits, other
    batches the same energy to the convergence target (1e-8 Eh)."""
    norb = n + 2
    h, eri, _ = ms.gen_integrals(norb, nsig, 67)
    ref = list(range(nsig))
    tk = np.array(list(itertools.islice(itertools.combinations(range(nsig, norb), n - nsig), 24)),
                  dtype=np.int32)

    def solve(max_batch):
        m = lib.MBE(0, precision=lib.MBE_MIXED_BF16X3, max_batch=max_batch)
        m.load(h, eri, 2 * nsig)
        lib.mbe_set_reference(m.ctx, ref, list(range(nsig, norb)))
        e, st = lib.mbe_solve_tuples(m.ctx, tk, n - nsig)
        m.close()
        assert np.all(st == 0)
        return e

    for b in (1, 5, 24):
        assert np.array_equal(solve(b), solve(b))
        assert np.abs(solve(b) - solve(24)).max() < 1e-8
