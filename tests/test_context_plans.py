"""Every length that has compile-time two-pass kernels is planned as those two passes
(CPU: the plans of the built library), so that no kernel is compiled for nothing and no
short axis falls to a one-pass kernel with an item a pencil."""
import ctypes as C

import pytest

from paper_2010_00409_gb300 import psatd


class Plan(C.Structure):
    _fields_ = [("N", C.c_int), ("npass", C.c_int), ("radix", C.c_int * 8), ("div_nb", C.c_uint * 8),
                ("div_l", C.c_uint * 8), ("div_run", C.c_uint)]


class Entry(C.Structure):
    _fields_ = [(n, C.c_int) for n in ("N", "R1", "cols_threads", "cols_smem", "rows_threads", "rows_per_block",
                                       "rows_smem", "kspace_threads", "kspace_smem")] + [
        ("cols", C.c_void_p * 2), ("rows", C.c_void_p * 2), ("kspace", C.c_void_p)]


def test_no_kernel_for_axes_that_always_take_another(plans):
    """x axes of 64, 128, 256 and 512 points and 512-point columns have register kernels
    of their own (fft_fast.cu, fft_three.cu): no two-pass kernel is compiled for them."""
    find = psatd.lib()["_ZN5psatd14two_pass_entryEi"]              # (a function object of its own)
    find.restype, find.argtypes = C.c_void_p, [C.c_int]
    entries = [Entry.from_address(find(n)) for n in range(1, 1025) if find(n)]
    for e in entries:
        assert bool(e.rows[0]) == bool(e.rows[1]) == (e.N not in (64, 128, 256, 512)), e.N
        assert bool(e.cols[0]) == bool(e.cols[1]) == (e.N * 16 * 8 < 96 * 1024 and e.N != 512), e.N


@pytest.fixture(scope="module")
def plans():
    lib = psatd.lib()
    plan, entry = lib._ZN5psatd12context_planEiiiPNS_8AxisPlanE, lib._ZN5psatd14two_pass_entryEi
    plan.restype, plan.argtypes = C.c_bool, [C.c_int, C.c_int, C.c_int, C.POINTER(Plan)]
    entry.restype, entry.argtypes = C.POINTER(C.c_int), [C.c_int]         # starts with N, R1

    def of(n, precision, axis=0):
        p = Plan()
        return list(p.radix[:p.npass]) if plan(n, precision, axis, C.byref(p)) else None

    def first_radix(n):
        e = entry(n)
        return e[1] if e else None
    return of, first_radix


def test_compile_time_lengths_take_two_passes(plans):
    of, first_radix = plans
    lengths = [n for n in range(1, 2049) if first_radix(n)]
    assert len(lengths) > 60
    for n in lengths:
        r = of(n, 32)
        assert len(r) == 2 and r[0] == first_radix(n) and r[0] * r[1] == n, (n, r)


def test_plans_multiply_to_their_length(plans):
    of, _ = plans
    for n in range(1, 2049):
        smooth = n
        for f in (2, 3, 5):
            while smooth % f == 0:
                smooth //= f
        for precision, axis, most in ((32, 0, 32), (32, 2, 32), (64, 0, 16), (64, 1, 16), (64, 2, 20)):
            r = of(n, precision, axis)
            assert (r is None) == (smooth != 1), n
            if r:
                product = 1
                for x in r:
                    product *= x
                assert product == n and max(r) <= most, (n, r)
