"""A context under a device-memory cap after a call that ran out of memory: the
tables of an active-space shape outlive the call, so a set of them left half
made must not be taken for a complete one by the next.

The cap is scanned in steps below the smallest table (20 links of 126 strings,
10,080 bytes), so that every allocation of the solve is the failing one for
some cap.  At each cap a solve that fails has to say MBE_ENOMEM, and a sigma
vector of the same shape, which needs a fraction of the memory, is right or
says MBE_ENOMEM too.
"""
import numpy as np
import pytest

import mbe_synth as ms
from oracle import casci as oc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_1905_02786_gb300 import build, _binding
    build.build()
    _binding.load_library()
    return _binding


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_sigma_after_failed_solve(lib, precision):
    prec = lib.MBE_FP64 if precision == "fp64" else lib.MBE_MIXED_BF16X3
    h, eri, _ = ms.gen_integrals(10, 4, 31)
    ref, exp, act = [0, 1, 2, 3], list(range(4, 10)), list(range(9))
    tuples = np.array([[4, 5, 6, 7, 8]], dtype=np.int32)        # 8e/9o
    c = ms.random_symmetric_ci(126, 3)[0]
    m = lib.MBE(0, precision=prec)
    m.load(h, eri, 8)
    want, _ = lib.mbe_sigma(m.ctx, act, c)
    m.close()
    e_or = oc.casci(h, eri, 4, act)
    failed_then_right = solved = 0
    for cap in range(96 << 10, 8 << 20, 8 << 10):
        m = lib.MBE(0, precision=prec, mem_cap_bytes=cap)
        failed = False
        try:
            m.load(h, eri, 8)
            lib.mbe_set_reference(m.ctx, ref, exp)
            eps, st = lib.mbe_solve_tuples(m.ctx, tuples, 5)
            assert st[0] == 0 and abs(eps[0] - e_or) < 1e-8
            solved += 1
        except lib.MBEError as err:
            assert err.code == lib.MBE_ENOMEM
            failed = True
        try:
            got, _ = lib.mbe_sigma(m.ctx, act, c)
            assert np.array_equal(got, want)
            failed_then_right += failed
        except lib.MBEError as err:
            assert failed and err.code in (lib.MBE_ENOMEM, lib.MBE_ESTATE)
        m.close()
        if solved >= 3:
            break
    assert solved and failed_then_right


@pytest.mark.parametrize("cap", [256, 512, 1024, 2048, 16 << 10, 24 << 10])
def test_no_integrals_after_failed_load(lib, cap):
    """10 orbitals take 1,024 and 24,320 bytes: none of these caps holds both."""
    h, eri, _ = ms.gen_integrals(10, 4, 31)
    m = lib.MBE(0, mem_cap_bytes=cap)
    with pytest.raises(lib.MBEError) as ei:
        m.load(h, eri, 8)
    assert ei.value.code == lib.MBE_ENOMEM
    for call in (lambda: lib.mbe_sigma(m.ctx, list(range(9)), np.ones(126 * 126)),
                 lambda: lib.mbe_set_reference(m.ctx, [3], [4, 5]),
                 lambda: lib.mbe_solve_tuples(m.ctx, np.array([[4]], dtype=np.int32), 1)):
        with pytest.raises(lib.MBEError) as ei:
            call()
        assert ei.value.code == lib.MBE_ESTATE
    m.close()


def test_increments_after_failed_growth(lib):
    """Order 2 of 64 expansion orbitals outgrows the tuple hash (4,096 slots for
    2,080 tuples): where the larger one does not fit, the call says so every
    time, and where it does the increments are right."""
    norb = 65
    rng = np.random.default_rng(4)
    h, eri, _ = ms.gen_integrals(norb, 1, 7)
    exp = list(range(1, norb))
    t1 = np.array([[o] for o in exp], dtype=np.int32)
    t2 = np.array([[a, b] for a in exp for b in exp if a < b], dtype=np.int32)
    e1, e2 = rng.standard_normal(len(t1)), rng.standard_normal(len(t2))
    base = eri.nbytes
    seen = set()
    for cap in range(base + (64 << 10), base + (2 << 20), 32 << 10):
        m = lib.MBE(0, mem_cap_bytes=cap)
        try:
            m.load(h, eri, 2)
            e0 = lib.mbe_set_reference(m.ctx, [0], exp)
            lib.mbe_set_order_energies(m.ctx, t1, e1, 1)
            inc1 = lib.mbe_increments(m.ctx, 1, 0.0, len(t1))[0]
            lib.mbe_set_order_energies(m.ctx, t2, e2, 2)
        except lib.MBEError as err:
            assert err.code == lib.MBE_ENOMEM
            m.close()
            continue
        want = e2 - e0 - inc1[t2[:, 0] - 1] - inc1[t2[:, 1] - 1]
        for _ in range(2):
            try:
                inc2 = lib.mbe_increments(m.ctx, 2, 0.0, len(t2))[0]
                assert np.abs(inc2 - want).max() < 1e-12
                seen.add("right")
                break
            except lib.MBEError as err:
                assert err.code == lib.MBE_ENOMEM
                seen.add("full")
        m.close()
    assert seen == {"right", "full"}


def test_no_order_after_failed_upload(lib):
    """The 2,016 tuples and energies of order 2 (16 KB each) that do not fit are
    not taken for a solved order."""
    norb = 65
    rng = np.random.default_rng(4)
    h, eri, _ = ms.gen_integrals(norb, 1, 7)
    exp = list(range(1, norb))
    t1 = np.array([[o] for o in exp], dtype=np.int32)
    t2 = np.array([[a, b] for a in exp for b in exp if a < b], dtype=np.int32)
    e1, e2 = rng.standard_normal(len(t1)), rng.standard_normal(len(t2))
    failed = 0
    for cap in range(eri.nbytes + (64 << 10), eri.nbytes + (512 << 10), 8 << 10):
        m = lib.MBE(0, mem_cap_bytes=cap)
        try:
            m.load(h, eri, 2)
            lib.mbe_set_reference(m.ctx, [0], exp)
            lib.mbe_set_order_energies(m.ctx, t1, e1, 1)
            lib.mbe_increments(m.ctx, 1, 0.0, len(t1))
        except lib.MBEError as err:
            assert err.code == lib.MBE_ENOMEM
            m.close()
            continue
        try:
            lib.mbe_set_order_energies(m.ctx, t2, e2, 2)
        except lib.MBEError as err:
            assert err.code == lib.MBE_ENOMEM
            failed += 1
            with pytest.raises(lib.MBEError) as ei:
                lib.mbe_increments(m.ctx, 2, 0.0, len(t2))
            assert ei.value.code == lib.MBE_ESTATE
        m.close()
    assert failed
