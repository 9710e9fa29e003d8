"""Every length that has compile-time two-pass kernels is planned as those two passes
(CPU: the plans of the built library), so that no kernel is compiled for nothing and no
short axis falls to a one-pass kernel with an item a pencil."""
import ctypes as C

import pytest

from paper_2010_00409_gb300 import psatd


class Plan(C.Structure):
    _fields_ = [("N", C.c_int), ("npass", C.c_int), ("radix", C.c_int * 8), ("div_nb", C.c_uint * 8),
                ("div_l", C.c_uint * 8), ("div_run", C.c_uint)]


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
