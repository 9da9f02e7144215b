"""mbe_sigma_noalloc where sigma overwrites c (the same buffer, or buffers that
overlap by a part): the same bits as with separate buffers.
"""
import math

import pytest

import mbe_synth as ms

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_1905_02786_gb300 import build, _binding
    build.build()
    _binding.load_library()
    return _binding


@pytest.mark.parametrize("nact,nocc", [(1, 1), (6, 3), (9, 4)])
@pytest.mark.parametrize("shift", [0.0, 0.5])
def test_in_place(lib, nact, nocc, shift):
    h, eri, _ = ms.gen_integrals(nact + 1, nocc, 6)
    act = list(range(nact))
    n = math.comb(nact, nocc) ** 2
    c = torch.tensor(ms.random_symmetric_ci(math.comb(nact, nocc), 30)[0].ravel(), device="cuda:0")
    m = lib.MBE(0, spin_shift=shift)
    m.load(h, eri, 2 * nocc)
    want = torch.empty_like(c)
    lib.mbe_sigma_noalloc(m.ctx, act, c, want)
    for off in (0, 1, n // 2, -(n // 3)):
        buf = torch.zeros(3 * n, dtype=torch.float64, device="cuda:0")
        buf[n:2 * n] = c
        out = buf[n + off:2 * n + off]
        torch.cuda.synchronize()
        lib.mbe_sigma_noalloc(m.ctx, act, buf[n:2 * n], out)
        assert torch.equal(out, want)
    m.close()
