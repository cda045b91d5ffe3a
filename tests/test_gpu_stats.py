"""gbcg_stats names the layout a handle's products run on, and counts the
bytes that layout reads."""
import numpy as np
import pytest
import scipy.sparse as sp

import femgen
import paper_1010_4639_gb300 as gb
from gpu_cases import fem

pytestmark = pytest.mark.gpu
ROWS, PLAN, TILES, DIAGONALS, UPPER_DIAGONALS = range(5)


@pytest.fixture(scope="module")
def torch():
    import torch
    gb.build()
    assert torch.cuda.is_available()
    return torch


def stats(fmt, arrays):
    with gb.Matrix(fmt, *arrays) as M:
        return M.stats()


@pytest.mark.parametrize("fmt", ["csr", "csc", "sym"])
def test_line_by_line_numbering(torch, fmt, monkeypatch):
    s = fem(17, 15, 19)
    n, nnz = s.n, s.nnz
    arrays = {"csr": (s.ptr, s.idx, s.val), "csc": s.csc(), "sym": s.upper()}[fmt]
    st = stats(fmt, arrays)
    held = 8 if fmt == "sym" else 15  # diagonals of linear tetrahedra on a box
    assert st["product"] == (UPPER_DIAGONALS if fmt == "sym" else DIAGONALS) and st["tiles"] == 0
    assert (st["spmv_bytes_fp64"], st["spmv_bytes_fp32"]) == (8 * held * n + 16 * n, 4 * held * n + 8 * n)
    assert st["layout"] == (2 if fmt == "sym" else 0)  # the family, as before
    monkeypatch.setenv("GBCG_DIAGONALS", "0")
    st = stats(fmt, arrays)
    if fmt == "sym":
        stored = (nnz + n) // 2
        assert st["product"] == TILES and st["tiles"] > 0
        assert st["spmv_bytes_fp64"] == 12 * stored + 4 * (n + 1) + 16 * n
        monkeypatch.setenv("GBCG_SYM_LAYOUT", "plan")
        assert stats(fmt, arrays)["product"] == PLAN
    else:
        assert st["product"] == ROWS and st["index_bytes"] == 2
        assert st["spmv_bytes_fp64"] == 10 * nnz + 4 * (n + 1) + 16 * n
        assert st["spmv_bytes_fp32"] == 6 * nnz + 4 * (n + 1) + 8 * n
        monkeypatch.setenv("GBCG_WIDE_INDEX", "1")
        st = stats(fmt, arrays)
        assert st["index_bytes"] == 4 and st["spmv_bytes_fp64"] == 12 * nnz + 4 * (n + 1) + 16 * n


def test_scattered_symmetric_storage_counts_both_copies(torch):
    s = fem(31, 31, 32)
    p = np.random.default_rng(3).permutation(s.n)
    A = sp.csr_matrix((s.val, s.idx, s.ptr), shape=(s.n, s.n))[p][:, p].tocsr()
    A.sort_indices()
    up = femgen.upper(s.n, A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data)
    st = stats("sym", up)
    assert st["product"] == ROWS and st["layout"] == 2 and st["index_bytes"] == 2
    assert st["spmv_bytes_fp32"] == 6 * s.nnz + 4 * (s.n + 1) + 8 * s.n
