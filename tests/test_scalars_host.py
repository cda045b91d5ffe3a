"""The solvers' scalar arithmetic on the CPU: the division (csrc/fp64.cuh) gives
the bits of the IEEE division over the whole range, and the fixed-point grid
sum (csrc/chip_solve.cuh) is as close to the exact sum as a rounding."""
import ctypes

import numpy as np
import pytest

import chip_check


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return chip_check.load(tmp_path_factory.mktemp("chip"))


def test_division_gives_the_ieee_quotient(lib):
    a, b = chip_check.dividends_and_divisors()
    q = np.empty_like(a)
    lib.host_div(chip_check.addr(a), chip_check.addr(b), chip_check.addr(q), ctypes.c_int64(a.size))
    with np.errstate(all="ignore"):
        ref = a / b
    assert chip_check.same(q, ref)


@pytest.mark.parametrize("G", [1, 7, 152, 255])
def test_fixed_point_sums(lib, G):
    parts, prevs = chip_check.sums(G)
    out = np.zeros(1)
    lib.host_fixed_sum.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_double, ctypes.c_void_p]
    taken = 0
    for part, prev in zip(parts, prevs):
        if not 1e-200 < prev < 1e200:
            continue  # such sums never take this form
        again = lib.host_fixed_sum(chip_check.addr(part), G, prev, chip_check.addr(out))
        assert again in (0, 1)
        if not again:
            chip_check.check_sum(part, prev, out[0], False)
            taken += 1
        else:  # as the solver does
            with np.errstate(invalid="ignore"):
                chip_check.check_sum(part, prev, part.sum(), True)
    assert taken > 200
