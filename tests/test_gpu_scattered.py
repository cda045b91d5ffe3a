"""Symmetric storage of matrices whose neighbours are scattered (computed from
the full operator's rows): products and solves against the oracle and against
the tiles, value updates, and row-gather solves with their vectors on the chip
(16- and 32-bit columns, empty and long rows, ragged ends)."""
import numpy as np
import pytest
import scipy.sparse as sp

import femgen
import oracle
import paper_1010_4639_gb300 as gb
from gpu_cases import fem, random_spd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch
    gb.build()
    assert torch.cuda.is_available()
    return torch


def scattered(grid, seed=3):
    """A finite-element matrix with its unknowns renumbered at random."""
    s = fem(*grid)
    p = np.random.default_rng(seed).permutation(s.n)
    A = sp.csr_matrix((s.val, s.idx, s.ptr), shape=(s.n, s.n))[p][:, p].tocsr()
    A.sort_indices()
    return s.n, A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data


@pytest.mark.parametrize("grid", [(12, 12, 12), (17, 15, 19), (31, 31, 32)])
def test_symmetric_products_and_updates(torch, grid, monkeypatch):
    n, ptr, idx, val = scattered(grid)
    up = femgen.upper(n, ptr, idx, val)
    x = femgen.random_vector(n, 4)
    xd, x32 = torch.from_numpy(x).cuda(), x.astype(np.float32)
    with gb.Matrix("sym", *up) as A:
        st = A.stats()
        assert st["layout"] == 2 and st["tiles"] == 0 and st["nnz_full"] == len(idx)
        assert st["stored_slots"] >= len(idx)
        y = A.spmv(xd).cpu().numpy()
        assert np.all(np.abs(y - oracle.spmv("sym", *up, x)) <= 1e-13 * oracle.abs_spmv("sym", *up, x))
        f = A.spmv_f32(torch.from_numpy(x32).cuda()).cpu().numpy()
        v32 = up[2].astype(np.float32)
        ref = oracle.spmv_f32("sym", up[0], up[1], v32, x32).astype(np.float64)
        scale = oracle.abs_spmv("sym", up[0], up[1], v32.astype(np.float64), x32.astype(np.float64))
        assert np.all(np.abs(f - ref) <= 1e-5 * scale)
        with pytest.raises(gb.GbcgError, match="row-gather"):
            A.solve(xd, variant="pipelined")
        new = up[2] * np.random.default_rng(1).uniform(0.5, 1.5, len(up[2]))
        A.update_values(torch.from_numpy(new).cuda())
        with gb.Matrix("sym", up[0], up[1], new) as F:
            assert torch.equal(A.spmv(xd), F.spmv(xd))
            assert torch.equal(A.spmv_f32(xd.float()), F.spmv_f32(xd.float()))
    monkeypatch.setenv("GBCG_SYM_LAYOUT", "tiles")
    with gb.Matrix("sym", *up) as T:
        assert T.stats()["tiles"] > 0
        assert np.all(np.abs(T.spmv(xd).cpu().numpy() - y) <= 2e-13 * oracle.abs_spmv("sym", *up, x))


@pytest.mark.parametrize("fmt,precision", [("csr", "fp64"), ("csr", "fp32_ru"), ("csr", "fp32_ir"), ("sym", "fp64"),
                                           ("sym", "fp32_ru"), ("csc", "fp64")])
@pytest.mark.parametrize("grid,ctas", [((12, 12, 12), None), ((31, 31, 32), None), ((17, 15, 19), "1"),
                                       ((31, 31, 32), "5")])
@pytest.mark.parametrize("wide", ["0", "1"])
def test_solves(torch, fmt, precision, grid, ctas, wide, monkeypatch):
    # 17 x 15 x 19 on one CTA and 31 x 31 x 32 on five reach both sides of the rows a CTA keeps on the chip
    n, ptr, idx, val = scattered(grid)
    if ctas:
        monkeypatch.setenv("GBCG_GRID", ctas)
    monkeypatch.setenv("GBCG_WIDE_INDEX", wide)
    arrays = femgen.upper(n, ptr, idx, val) if fmt == "sym" else (ptr, idx, val)
    xs = femgen.random_vector(n, 8)
    b = oracle.spmv("csr", ptr, idx, val, xs)
    with gb.Matrix(fmt, *arrays) as A:
        x, info = A.solve(torch.from_numpy(b).cuda(), tol=1e-11, maxit=10 * n, precision=precision)
        again, _ = A.solve(torch.from_numpy(b).cuda(), tol=1e-11, maxit=10 * n, precision=precision)
    assert info.status == "OK" and torch.equal(x, again)
    r = b - oracle.spmv("csr", ptr, idx, val, x.cpu().numpy())
    assert np.linalg.norm(r) <= 1e-11 * np.linalg.norm(b)


@pytest.mark.parametrize("precision", ["fp64", "fp32_ru"])
def test_long_rows_on_the_chip(torch, precision):
    ptr, idx, val = random_spd(2999, 9, density=0.003, dense_rows=(7, 1500, 2998))
    b = np.random.default_rng(1).uniform(-1, 1, 2999)
    ref = oracle.cg("csr", ptr, idx, val, b, tol=1e-12)
    with gb.Matrix("csr", ptr, idx, val) as A:
        assert A.stats()["long_rows"] >= 1
        x, info = A.solve(torch.from_numpy(b).cuda(), tol=1e-12, precision=precision)
    assert info.status == "OK"
    assert np.linalg.norm(x.cpu().numpy() - ref.x) <= 1e-8 * np.linalg.norm(ref.x)
