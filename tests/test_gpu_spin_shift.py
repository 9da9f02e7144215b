"""Mixed-precision sigma vectors with a spin shift against the FP64 mode: the
shift must not add to the error.  The split of g' and c into two BF16 parts
gives the rms error at shift 0; the spin term in FP32 adds about
|shift| (nsig^2 + nsig) 2^-24 of rms c (its terms times one rounding each) to it,
and 10 % are left for shifts that go through the split operand.
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


@pytest.mark.parametrize("n,nsig", [(9, 4), (10, 5), (12, 4), (9, 6), (13, 3)])
def test_error_independent_of_shift(lib, n, nsig):
    nstr = len(list(itertools.combinations(range(n), nsig)))
    sq = {}
    for seed in range(4):
        h, eri, _ = ms.gen_integrals(n, nsig, 300 + seed)
        c = ms.random_symmetric_ci(nstr, seed)[0].astype(np.float32).astype(np.float64)
        for shift in (0.0, 0.25, 0.5, 1.0, 4.0, 64.0, -2.0):
            sig = []
            for prec in (lib.MBE_FP64, lib.MBE_MIXED_BF16X3):
                m = lib.MBE(0, precision=prec, spin_shift=shift)
                m.load(h, eri, 2 * nsig)
                sig.append(lib.mbe_sigma(m.ctx, list(range(n)), c)[0])
                m.close()
            sq.setdefault(shift, []).append(np.mean((sig[1] - sig[0]) ** 2) / np.mean(c ** 2))
    rms = {s: np.sqrt(np.mean(v)) for s, v in sq.items()}
    for shift, r in rms.items():
        assert r <= 1.1 * rms[0.0] + abs(shift) * (nsig * nsig + nsig) * 2.0 ** -24, (shift, rms)
