"""The solvers' scalar division (csrc/fp64.cuh) on the CPU: the bits of the
IEEE division over the whole range."""
import numpy as np
import pytest

import chip_check


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return chip_check.load(tmp_path_factory.mktemp("chip"))


def test_division_gives_the_ieee_quotient(lib):
    a, b = chip_check.dividends_and_divisors()
    q = np.empty_like(a)
    lib.host_div(chip_check.addr(a), chip_check.addr(b), chip_check.addr(q), chip_check.ctypes.c_int64(a.size))
    with np.errstate(all="ignore"):
        ref = a / b
    assert chip_check.same(q, ref)
