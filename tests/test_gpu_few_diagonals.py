"""Every number of diagonals from 1 to 18, so that the product's last chunk has
every size in every precision and kernel (one-shot, on the chip, vectors in
memory): products against the oracle (|y - y_oracle| <= 1e-13 (|A||x|), in single precision
1e-5) and, in full storage, bit for bit against the row gather, which sums in
the same order; solves to 1e-12.  And the time of a matrix of two or three
stored diagonals against the same matrix in tiles."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle
import paper_1010_4639_gb300 as gb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch
    gb.build()
    assert torch.cuda.is_available()
    return torch


def spd(n, upper_offsets, seed):
    """A diagonally dominant symmetric matrix with these diagonals above the main one."""
    rng = np.random.default_rng(seed)
    U = sp.diags([-rng.uniform(0.1, 1.0, n - o) for o in upper_offsets], upper_offsets, shape=(n, n), format="csr") \
        if upper_offsets else sp.csr_matrix((n, n))
    A = U + U.T
    A = (A + sp.diags(-np.asarray(A.sum(axis=1)).ravel() + 0.1)).tocsr()
    A.sort_indices()
    return A


def arrays(A, fmt):
    M = sp.triu(A).tocsr() if fmt == "sym" else A
    M.sort_indices()
    return M.indptr.astype(np.int32), M.indices.astype(np.int32), M.data


def both(fmt, arrs, monkeypatch):
    D = gb.Matrix(fmt, *arrs)
    monkeypatch.setenv("GBCG_DIAGONALS", "0")
    O = gb.Matrix(fmt, *arrs)
    monkeypatch.delenv("GBCG_DIAGONALS")
    return D, O


OFFSETS = [1, 2, 3, 5, 8, 40, 41, 42, 43, 200, 201, 202, 300, 301, 302, 303, 304]


@pytest.mark.parametrize("above", range(18))
@pytest.mark.parametrize("fmt,extra", [("csr", 0), ("csr", 1), ("sym", 0)])
def test_products(torch, above, fmt, extra, monkeypatch):
    # extra: one more diagonal below, so that full storage holds even numbers of them too
    n = 3001
    offs = OFFSETS[:above]
    A = spd(n, offs, above)
    if fmt == "csr":
        A = sp.triu(A, -min(above, 1) * 3).tocsr() if above else A  # above the main diagonal, and a few below
        if extra:
            A = (A + sp.diags(np.full(n - 7, 0.5), -7, shape=(n, n))).tocsr()
    arrs = arrays(A, fmt)
    x = np.random.default_rng(1).uniform(-1, 1, n)
    x32, v32 = x.astype(np.float32), arrs[2].astype(np.float32)
    D, O = both(fmt, arrs, monkeypatch)
    with D, O:
        yd, yo = (M.spmv(torch.from_numpy(x).cuda()).cpu().numpy() for M in (D, O))
        fd, fo = (M.spmv_f32(torch.from_numpy(x32).cuda()).cpu().numpy() for M in (D, O))
    assert np.all(np.abs(yd - oracle.spmv(fmt, *arrs, x)) <= 1e-13 * oracle.abs_spmv(fmt, *arrs, x))
    ref = oracle.spmv_f32(fmt, arrs[0], arrs[1], v32, x32).astype(np.float64)
    scale = oracle.abs_spmv(fmt, arrs[0], arrs[1], v32.astype(np.float64), x32.astype(np.float64))
    assert np.all(np.abs(fd - ref) <= 1e-5 * scale)
    if fmt == "csr":
        assert np.array_equal(yd, yo) and np.array_equal(fd, fo)


@pytest.mark.parametrize("above", [0, 1, 2, 3, 4, 5, 8, 9, 16])
@pytest.mark.parametrize("fmt", ["csr", "sym"])
@pytest.mark.parametrize("ctas", [None, "5", "1"])
def test_solves(torch, above, fmt, ctas, monkeypatch):
    # 9 001 rows: one per thread on every SM, several on five CTAs, too many for the chip on one
    n = 9001
    if ctas:
        monkeypatch.setenv("GBCG_GRID", ctas)
    A = spd(n, OFFSETS[:above], 7 + above)
    b = A @ np.random.default_rng(2).uniform(-1, 1, n)
    with gb.Matrix(fmt, *arrays(A, fmt)) as M:
        for precision in ("fp64", "fp32_ru", "fp32_ir"):
            x, info = M.solve(torch.from_numpy(b).cuda(), tol=1e-12, maxit=10 * n, precision=precision)
            assert info.status == "OK", (precision, info)
            assert np.linalg.norm(b - A @ x.cpu().numpy()) <= 1.01e-12 * np.linalg.norm(b)


@pytest.mark.parametrize("offsets", [[1], [1, 1500]])
def test_two_and_three_stored_diagonals_are_not_slower_than_tiles(torch, offsets, monkeypatch):
    # 2.0 M rows, double precision, where whole chunks of eight took 58 us for a
    # product (tiles 41 and 50) and 84 us per iteration (tiles 70 and 78); a
    # tenth is allowed for what runs of one side differ by
    n = 2_000_000
    A = spd(n, offsets, 3)
    x = torch.rand(n, device="cuda", dtype=torch.float64)
    y = torch.empty_like(x)
    D, O = both("sym", arrays(A, "sym"), monkeypatch)
    best = {}
    with D, O:
        for M in (D, O):
            times, its = [], []
            for _ in range(5):
                M.spmv(x, y)
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                for _ in range(20):
                    M.spmv(x, y)
                b.record()
                torch.cuda.synchronize()
                times.append(a.elapsed_time(b) / 20)
                _, info = M.solve(x, tol=1e-30, maxit=100, raise_on_error=False)
                its.append(info.kernel_ms / info.iterations)
            best[M] = (min(times), min(its))
    assert best[D][0] <= 1.1 * best[O][0] and best[D][1] <= 1.1 * best[O][1], best
