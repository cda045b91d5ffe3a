"""The solvers' scalar arithmetic (csrc/fp64.cuh) and the on-chip solvers' grid
sums (csrc/chip_solve.cuh) on the GPU against IEEE results and exact sums: division and widening bit for bit, the finite, positive and
square-root tests by their outcome.  The square-root test may differ from
sqrt(s) <= c only where both sides agree to 1e-12, and there it takes the exact
test, so the outcomes are equal everywhere."""
import ctypes

import numpy as np
import pytest

import chip_check
import paper_1010_4639_gb300 as gb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch
    gb.build()
    assert torch.cuda.is_available()
    return torch


@pytest.fixture(scope="module")
def lib(tmp_path_factory, torch):
    return chip_check.load(tmp_path_factory.mktemp("chip"))


def call(f, *arrays):
    assert f(*[chip_check.addr(a) for a in arrays], ctypes.c_int64(arrays[0].numel())) == 0


def test_division_gives_the_ieee_quotient(torch, lib):
    a, b = chip_check.dividends_and_divisors()
    q = torch.empty(a.size, dtype=torch.float64, device="cuda")
    call(lib.gpu_div, torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), q)
    with np.errstate(all="ignore"):
        ref = a / b
    assert chip_check.same(q.cpu().numpy(), ref)


def test_widening_keeps_every_bit(torch, lib):
    f = np.random.default_rng(1).integers(0, 1 << 32, 1 << 20, dtype=np.uint64).astype(np.uint32).view(np.float32)
    f = np.concatenate([f, np.array([0, -0.0, 1e-45, -1e-45, 1.1754944e-38, 3.4028235e38, np.inf, -np.inf, np.nan],
                                    np.float32)])
    d = torch.empty(f.size, dtype=torch.float64, device="cuda")
    call(lib.gpu_widen, torch.from_numpy(f).cuda(), d)
    with np.errstate(invalid="ignore"):  # signalling NaNs
        assert chip_check.same(d.cpu().numpy(), f.astype(np.float64))


def test_tests_of_a_sum(torch, lib):
    rng = np.random.default_rng(2)
    c = 10.0 ** rng.uniform(-170, 170, 1 << 18)
    with np.errstate(over="ignore", under="ignore"):
        s = c * c * (1.0 + rng.choice([0.0, 1e-16, -3e-16, 1e-13, -1e-13, 3e-12, -3e-12, 0.5, -0.5], c.size))
    special = np.array([0.0, 5e-324, 1e-300, 1.0, 1e300, np.inf, np.nan])
    s2, c2 = (x.ravel() for x in np.meshgrid(special, special))
    s, c = np.concatenate([s, s2]), np.concatenate([c, c2])
    out = torch.empty(s.size, dtype=torch.int32, device="cuda")
    call(lib.gpu_tests, torch.from_numpy(s).cuda(), torch.from_numpy(c).cuda(), out)
    out = out.cpu().numpy()
    assert np.array_equal((out & 1) != 0, np.isfinite(s))
    ok = np.isfinite(s)
    assert np.array_equal((out[ok] & 2) != 0, s[ok] > 0)
    assert np.array_equal((out & 4) != 0, (out & 8) != 0)
    with np.errstate(invalid="ignore"):
        assert np.array_equal((out & 8) != 0, np.sqrt(s) <= c)


def grid_sums(torch, lib, parts, prevs, absent=-1, timeout_ms=1000):
    cases, G = parts.shape
    out = torch.zeros((cases, G), dtype=torch.float64, device="cuda")
    retaken = torch.full((cases, G), -1, dtype=torch.int32, device="cuda")
    ok = torch.full((cases, G), -1, dtype=torch.int32, device="cuda")
    status = np.zeros(1, np.int32)
    a = [chip_check.addr(t) for t in (torch.from_numpy(parts).cuda(), torch.from_numpy(prevs).cuda(), out, retaken, ok)]
    rc = lib.gpu_sums(*a, cases, G, absent, timeout_ms, chip_check.addr(status))
    assert rc == 0
    return out.cpu().numpy(), retaken.cpu().numpy(), ok.cpu().numpy(), int(status[0])


@pytest.mark.parametrize("G", [1, 7, 152])
def test_grid_sums(torch, lib, G):
    parts, prevs = chip_check.sums(G)
    out, retaken, ok, status = grid_sums(torch, lib, parts, prevs)
    assert status == 0 and np.all(ok == 1)
    for i in range(len(prevs)):
        assert chip_check.same(out[i], np.full(G, out[i, 0])) and np.all(retaken[i] == retaken[i, 0])
        if not 1e-200 < prevs[i] < 1e200:
            assert retaken[i, 0] == 1  # the earlier sum's exponent is out of the fixed point's range
        chip_check.check_sum(parts[i], prevs[i], out[i, 0], retaken[i, 0] == 1)


@pytest.mark.parametrize("prev", [1.0, 0.0])
def test_a_grid_sums_wait_ends(torch, lib, prev):
    # a CTA that never arrives: both forms of the sum give up within their limit
    _, _, ok, status = grid_sums(torch, lib, np.ones((1, 5)), np.array([prev]), absent=0, timeout_ms=20)
    assert status == 5 and list(ok[0]) == [-1, 0, 0, 0, 0]
    # and the device is as before
    out, _, ok, status = grid_sums(torch, lib, np.ones((1, 5)), np.array([prev]))
    assert status == 0 and np.all(ok == 1) and np.all(out == 5.0)
