"""Products and solves on the diagonal layout against the oracle, and against
the layouts the same matrices take without it (GBCG_DIAGONALS=0): tile edges
of the thread blocks, rows whose columns leave the matrix, non-symmetric
values, non-finite vector elements and value updates.

Double precision: |y - y_oracle| <= 1e-13 (|A||x|); single: 1e-5 (|A32||x|).
Full storage sums a row in the row-gather layout's order, so there the two
layouts agree bit for bit."""
import numpy as np
import pytest
import scipy.sparse as sp

import femgen
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


def banded(n, offsets, seed):
    rng = np.random.default_rng(seed)
    rows = np.repeat(np.arange(n), len(offsets))
    cols = rows + np.tile(offsets, n)
    ok = (cols >= 0) & (cols < n)
    A = sp.csr_matrix((rng.uniform(-1, 1, ok.sum()), (rows[ok], cols[ok])), shape=(n, n))
    A.sort_indices()
    return A


def both(fmt, arrays, monkeypatch):
    D = gb.Matrix(fmt, *arrays)
    monkeypatch.setenv("GBCG_DIAGONALS", "0")
    O = gb.Matrix(fmt, *arrays)
    monkeypatch.delenv("GBCG_DIAGONALS")
    return D, O


@pytest.mark.parametrize("n,offsets", [(1, [0]), (31, [0, 1]), (256, [-1, 0, 1]), (257, [-200, 0, 200]),
                                       (1000, [-128, -33, -1, 0, 1, 32, 40, 64, 500]), (5000, list(range(-12, 20)))])
@pytest.mark.parametrize("fmt", ["csr", "sym", "csc"])
def test_products(torch, n, offsets, fmt, monkeypatch):
    A = banded(n, offsets, n)
    if fmt == "sym":
        A = sp.triu(A + A.T).tocsr()
    elif fmt == "csc":
        A = A.tocsc()
    A.sort_indices()
    arrays = (A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data)
    x = np.random.default_rng(5).uniform(-1, 1, n)
    x32 = x.astype(np.float32)
    v32 = arrays[2].astype(np.float32)
    D, O = both(fmt, arrays, monkeypatch)
    with D, O:
        yd, yo = (M.spmv(torch.from_numpy(x).cuda()).cpu().numpy() for M in (D, O))
        fd, fo = (M.spmv_f32(torch.from_numpy(x32).cuda()).cpu().numpy() for M in (D, O))
    assert np.all(np.abs(yd - oracle.spmv(fmt, *arrays, x)) <= 1e-13 * oracle.abs_spmv(fmt, *arrays, x))
    ref = oracle.spmv_f32(fmt, arrays[0], arrays[1], v32, x32).astype(np.float64)
    scale = oracle.abs_spmv(fmt, arrays[0], arrays[1], v32.astype(np.float64), x32.astype(np.float64))
    assert np.all(np.abs(fd - ref) <= 1e-5 * scale)
    if fmt != "sym":
        assert np.array_equal(yd, yo) and np.array_equal(fd, fo)


@pytest.mark.parametrize("fmt", ["csr", "csc"])
def test_non_finite_elements_reach_only_their_rows(torch, fmt, monkeypatch):
    s = fem(9, 10, 11)
    x = torch.from_numpy(femgen.random_vector(s.n, 6)).cuda()
    x[100], x[400], x[500] = float("inf"), float("-inf"), float("nan")
    D, O = both(fmt, (s.ptr, s.idx, s.val), monkeypatch)
    with D, O:
        for y, z in ((D.spmv(x), O.spmv(x)), (D.spmv_f32(x.float()), O.spmv_f32(x.float()))):
            rows = np.repeat(np.arange(s.n), np.diff(s.ptr))
            hit = np.zeros(s.n, bool)
            hit[rows[np.isin(s.idx, [100, 400, 500])]] = True
            assert np.array_equal(~np.isfinite(y.cpu().numpy()), hit)
            ok = torch.from_numpy(~hit).cuda()
            assert torch.equal(y[ok], z[ok])


@pytest.mark.parametrize("fmt", ["csr", "sym"])
def test_value_updates_keep_zeros_and_padding(torch, fmt, monkeypatch):
    # stored zeros of either sign and values below single precision's range stay entries
    s = fem(9, 10, 11)
    arrays = (s.ptr, s.idx, s.val) if fmt == "csr" else s.upper()
    new = arrays[2].copy()
    new[::7], new[1::7], new[2::7] = 0.0, -0.0, -1e-60
    x = torch.from_numpy(femgen.random_vector(s.n, 8)).cuda()
    with gb.Matrix(fmt, *arrays) as A, gb.Matrix(fmt, arrays[0], arrays[1], new) as F:
        A.update_values(torch.from_numpy(new).cuda())
        assert torch.equal(A.spmv(x), F.spmv(x)) and torch.equal(A.spmv_f32(x.float()), F.spmv_f32(x.float()))
        x[:] = float("inf")
        y = A.spmv_f32(x.float())
        assert torch.isnan(y).any() and torch.equal(torch.isnan(y), torch.isnan(F.spmv_f32(x.float())))


@pytest.mark.parametrize("fmt,precision", [("csr", "fp64"), ("csr", "fp32_ru"), ("csr", "fp32_ir"), ("sym", "fp64"),
                                           ("sym", "fp32_ru"), ("sym", "fp32_ir"), ("csc", "fp32_ru")])
# few rows per CTA; several product steps per thread; the vectors of a CTA too
# large for the chip (25 230 rows on one CTA); ragged last slices throughout
@pytest.mark.parametrize("grid,ctas", [((31, 31, 32), None), ((17, 15, 19), "7"), ((12, 12, 12), "1"),
                                       ((31, 31, 32), "9"), ((31, 31, 32), "1")])
def test_solves(torch, fmt, precision, grid, ctas, monkeypatch):
    s = fem(*grid)
    if ctas:
        monkeypatch.setenv("GBCG_GRID", ctas)
    arrays = s.upper() if fmt == "sym" else (s.ptr, s.idx, s.val)
    b = torch.from_numpy(s.b).cuda()
    D, O = both(fmt, arrays, monkeypatch)
    with D, O:
        x, i = D.solve(b, tol=1e-12, maxit=10 * s.n, precision=precision)
        z, j = O.solve(b, tol=1e-12, maxit=10 * s.n, precision=precision)
        again, _ = D.solve(b, tol=1e-12, maxit=10 * s.n, precision=precision)
    assert i.status == j.status == "OK"
    assert torch.equal(x, again)
    r = s.b - oracle.spmv("csr", s.ptr, s.idx, s.val, x.cpu().numpy())
    assert np.linalg.norm(r) <= 1e-12 * np.linalg.norm(s.b)
    slack = 0.05 if precision == "fp64" else 0.1
    assert abs(i.iterations - j.iterations) <= 2 * (slack * j.iterations + 10)
    assert torch.linalg.norm(x - z) <= 1e-8 * torch.linalg.norm(z)


@pytest.mark.parametrize("precision", ["fp64", "fp32_ru", "fp32_ir"])
def test_tiles_asked_for_by_name(torch, precision, monkeypatch):
    # the tiled symmetric layout stays what irregular meshes take
    monkeypatch.setenv("GBCG_SYM_LAYOUT", "tiles")
    s = fem(17, 15, 19)
    with gb.Matrix("sym", *s.upper()) as A:
        assert A.stats()["tiles"] > 0
        x, info = A.solve(torch.from_numpy(s.b).cuda(), tol=1e-10, maxit=10 * s.n, precision=precision)
    assert info.status == "OK"
    r = s.b - oracle.spmv("csr", s.ptr, s.idx, s.val, x.cpu().numpy())
    assert np.linalg.norm(r) <= 1e-10 * np.linalg.norm(s.b)


@pytest.mark.parametrize("precision", ["fp32_ru", "fp32_ir", "fp64"])
@pytest.mark.parametrize("nrhs", [8, 3])
def test_batch(torch, precision, nrhs, monkeypatch):
    # instances on diagonals beside one that has too many (a random matrix) and
    # a tiny one turned down for its padding, against the same batch in CSR
    rng = np.random.default_rng(4)
    R = sp.random(300, 300, 0.02, random_state=4, format="csr")
    R = (R + R.T + sp.diags(np.full(300, 12.0))).tocsr()
    R.sort_indices()
    mats = [sp.csr_matrix((s.val, s.idx, s.ptr), shape=(s.n, s.n)) for s in
            (fem(9, 10, 11), fem(5, 5, 4), fem(14, 13, 12, seed_mesh=3), fem(20, 4, 9, contrast=10.0))]
    mats.insert(1, R)
    A = sp.block_diag(mats, format="csr")
    A.sort_indices()
    off = np.concatenate([[0], np.cumsum([m.shape[0] for m in mats])]).astype(np.int64)
    b = torch.from_numpy(np.ascontiguousarray(rng.uniform(-1, 1, (A.shape[0], nrhs)))).cuda()
    args = (off, A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data)
    out = []
    for flag in ("1", "0"):
        monkeypatch.setenv("GBCG_DIAGONALS", flag)
        with gb.Batch(*args, nrhs=nrhs, tune=False) as B:
            x, infos, rep = B.solve(b, tol=1e-12, maxit=20000, precision=precision)
            again, _, _ = B.solve(b, tol=1e-12, maxit=20000, precision=precision)
        assert rep["status"] == "OK" and torch.equal(x, again)
        r = b.cpu().numpy() - A @ x.cpu().numpy()
        for a, z in zip(off[:-1], off[1:]):
            bb = np.linalg.norm(b[a:z].cpu().numpy(), axis=0)
            assert np.all(np.linalg.norm(r[a:z], axis=0) <= 1.001e-12 * bb)
        out.append(x)
    assert torch.linalg.norm(out[0] - out[1]) <= 1e-8 * torch.linalg.norm(out[1])
