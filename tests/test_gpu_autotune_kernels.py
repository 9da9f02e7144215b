"""The autotuner's cache where a shape can take either two-spin kernel: each has
entries of its own ("sigma_ab n nsig ..." over the rows of c, nsig negated over
(N-1)-electron strings), plans of one are not taken for the other, and tuned runs
give the bits of untuned ones.  Also the kernel over the rows of c beyond 12
orbitals: its tuner, and its bounded waits.
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


def _solve(lib, n, nsig, count, **opts):
    norb = n + 2
    h, eri, _ = ms.gen_integrals(norb, nsig, 59)
    ref = list(range(nsig))
    tk = list(itertools.islice(itertools.combinations(range(nsig, norb), n - nsig), count))
    m = lib.MBE(0, precision=lib.MBE_MIXED_BF16X3, **opts)
    m.load(h, eri, 2 * nsig)
    lib.mbe_set_reference(m.ctx, ref, [p for p in range(norb) if p not in ref])
    eps, st = lib.mbe_solve_tuples(m.ctx, np.array(tk, dtype=np.int32), n - nsig)
    m.close()
    assert np.all(st == 0)
    return eps


# (shape, tuples, sign of nsig in the entry): less and more than half full, both
# sides of the least work per SM, beyond 12 orbitals
@pytest.mark.parametrize("n,nsig,count,sign", [
    (10, 4, 28, -1), (10, 4, 2, 1), (12, 5, 1, -1), (12, 9, 8, 1), (11, 7, 8, 1), (13, 3, 2, 1),
])
def test_entries_and_bits(lib, tmp_path, n, nsig, count, sign):
    cache = tmp_path / "tune.txt"
    # an entry of the other kernel for the same shape, with a plan that fits
    other = f"sigma_ab {n} {-sign * nsig} 2 0 1 0.001"
    cache.write_text(other + "\n")
    plain = _solve(lib, n, nsig, count)
    tuned = _solve(lib, n, nsig, count, autotune=1, tune_file=str(cache).encode())
    assert np.array_equal(plain, tuned)
    lines = [ln.split() for ln in cache.read_text().splitlines()]
    assert " ".join(lines[0]) == other
    assert [int(ln[2]) for ln in lines[1:] if int(ln[1]) == n] == [sign * nsig]
    again = _solve(lib, n, nsig, count, autotune=1, tune_file=str(cache).encode())
    assert np.array_equal(plain, again)
    assert len(cache.read_text().splitlines()) == len(lines)


def test_bounded_wait_beyond_12_orbitals(lib):
    n, nsig = 13, 3
    h, eri, _ = ms.gen_integrals(n, nsig, 59)
    c = ms.random_symmetric_ci(286, 3)[0]
    m = lib.MBE(0, precision=lib.MBE_MIXED_BF16X3, wait_limit=0)
    m.load(h, eri, 2 * nsig)
    with pytest.raises(lib.MBEError) as ei:
        lib.mbe_sigma(m.ctx, list(range(n)), c)
    assert ei.value.code == lib.MBE_ETIMEOUT
    m.close()
    sig = []
    for prec in (lib.MBE_FP64, lib.MBE_MIXED_BF16X3):
        m = lib.MBE(0, precision=prec)
        m.load(h, eri, 2 * nsig)
        sig.append(lib.mbe_sigma(m.ctx, list(range(n)), c)[0])
        m.close()
    assert np.abs(sig[1] - sig[0]).max() <= 2e-4 * np.abs(sig[0]).max()
