"""Solves whose sums leave the range of the on-chip solvers' fast forms: r'r that
falls to zero or by many orders in one step (the sum is taken again), and
right-hand sides so small or large that the sums' exponents lie outside the
fixed point's range and near the ends of the division's and the square-root
test's.  Double-precision CG does not depend on the scale of b: the count stays within
5% + 5 of the unscaled one."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle
import paper_1010_4639_gb300 as gb
from gpu_cases import fem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch
    gb.build()
    assert torch.cuda.is_available()
    return torch


def csr(A):
    A = A.tocsr()
    A.sort_indices()
    return A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data


@pytest.mark.parametrize("precision", ["fp64", "fp32_ru", "fp32_ir"])
@pytest.mark.parametrize("fmt", ["csr", "sym"])
def test_residual_falls_to_nothing_in_one_step(torch, precision, fmt):
    n = 7001
    b = np.random.default_rng(1).uniform(-1, 1, n)
    with gb.Matrix(fmt, *csr(sp.identity(n))) as A:
        x, info = A.solve(torch.from_numpy(b).cuda(), tol=1e-13, precision=precision)
    assert info.status == "OK" and info.iterations <= 3
    assert np.linalg.norm(x.cpu().numpy() - b) <= 1e-13 * np.linalg.norm(b)
    # two clusters of eigenvalues: the second step takes the residual down by some ten orders
    d = np.where(np.arange(n) % 2, 1.0, 1000.0)
    with gb.Matrix(fmt, *csr(sp.diags(d))) as A:
        x, info = A.solve(torch.from_numpy(b).cuda(), tol=1e-13, precision=precision)
    assert info.status == "OK" and info.iterations <= 10
    assert np.linalg.norm(b - d * x.cpu().numpy()) <= 1.001e-13 * np.linalg.norm(b)


@pytest.mark.parametrize("scale", [1e-140, 1e-125, 1e-60, 1e60, 1e125, 1e140])
@pytest.mark.parametrize("fmt", ["csr", "sym"])
@pytest.mark.parametrize("diagonals", ["1", "0"])
def test_scaled_right_hand_sides(torch, scale, fmt, diagonals, monkeypatch):
    monkeypatch.setenv("GBCG_DIAGONALS", diagonals)
    s = fem(17, 15, 19)
    arrays = s.upper() if fmt == "sym" else (s.ptr, s.idx, s.val)
    with gb.Matrix(fmt, *arrays) as A:
        x, info = A.solve(torch.from_numpy(s.b).cuda(), tol=1e-10, maxit=10 * s.n)
        y, scaled = A.solve(torch.from_numpy(s.b * scale).cuda(), tol=1e-10, maxit=10 * s.n)
    assert info.status == scaled.status == "OK"
    assert abs(info.iterations - scaled.iterations) <= 0.05 * info.iterations + 5
    r = s.b - oracle.spmv("csr", s.ptr, s.idx, s.val, y.cpu().numpy() / scale)
    assert np.linalg.norm(r) <= 1.001e-10 * np.linalg.norm(s.b)
