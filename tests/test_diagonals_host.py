"""The diagonal layout (csrc/layout.cpp, build_diagonals) on the CPU: which
matrices it takes, where every entry lands, and the kernels' row sums against
the general row-by-row product, over formats, index bases, ragged sizes,
missing diagonals, stored zeros and non-finite vector elements."""
import os
import struct
import subprocess

import numpy as np
import pytest
import scipy.sparse as sp

import femgen

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1010_4639_gb300", "csrc")
FORMAT = {"csr": 0, "sym": 1, "csc": 2}


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("dia") / "diagonals_check")
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", os.path.join(HERE, "diagonals_check.cpp"),
                    os.path.join(CSRC, "layout.cpp"), "-o", out], check=True)
    return out


def run(checker, tmp_path, fmt, arrays, x, base=0):
    ptr, idx, val = (np.asarray(a) for a in arrays)
    src, dst = str(tmp_path / "m.bin"), str(tmp_path / "y.bin")
    with open(src, "wb") as f:
        f.write(struct.pack("<qq", ptr.shape[0] - 1, idx.shape[0]))
        for a, t in ((ptr + base, np.int32), (idx + base, np.int32), (val, np.float64), (x, np.float64)):
            f.write(np.ascontiguousarray(a, dtype=t).tobytes())
    out = subprocess.run([checker, src, str(FORMAT[fmt]), str(base), dst], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
    word = out.stdout.split()[0]
    return word, np.fromfile(dst) if word == "OK" else None


def banded(n, offsets, seed, holes=0.0):
    """CSR of a random matrix on the given diagonals, a share of entries left out."""
    rng = np.random.default_rng(seed)
    rows = np.repeat(np.arange(n), len(offsets))
    cols = rows + np.tile(offsets, n)
    ok = (cols >= 0) & (cols < n) & (rng.random(rows.size) >= holes)
    A = sp.csr_matrix((rng.uniform(-1, 1, ok.sum()), (rows[ok], cols[ok])), shape=(n, n))
    A.sort_indices()
    return A


def arrays_of(A, fmt):
    if fmt == "csc":
        A = A.tocsc()
    elif fmt == "sym":
        A = sp.triu(A + A.T).tocsr()
    A.sort_indices()
    return A.indptr, A.indices, A.data


def reference(A, x, fmt):
    """Row sums over the stored entries only (inf and NaN as the general path meets them)."""
    if fmt == "sym":
        U = sp.triu(A + A.T).tocsr()
        A = U + sp.triu(U, 1).T
    A = A.tocsr()
    with np.errstate(invalid="ignore"):
        terms = A.data * x[A.indices]
        y = np.array([terms[a:b].sum() for a, b in zip(A.indptr[:-1], A.indptr[1:])])
        scale = np.array([np.abs(terms[a:b]).sum() for a, b in zip(A.indptr[:-1], A.indptr[1:])])
    return y, scale


def same(y, ref, scale):
    bad = ~np.isfinite(ref)
    assert np.array_equal(np.isnan(y), np.isnan(ref))
    assert np.array_equal(y[bad & ~np.isnan(ref)], ref[bad & ~np.isnan(ref)])
    assert np.all(np.abs(y[~bad] - ref[~bad]) <= 1e-14 * scale[~bad])


@pytest.mark.parametrize("fmt", ["csr", "sym", "csc"])
@pytest.mark.parametrize("n,offsets", [(1, [0]), (2, [0, 1]), (33, [-1, 0, 1]), (64, [0]), (200, [-17, -3, 0, 2, 5]),
                                       (1000, [-100, -10, -9, -1, 0, 1, 9, 10, 100]), (65, [3]), (65, [-3]),
                                       (4097, list(range(-15, 17)))])
@pytest.mark.parametrize("base", [0, 1])
def test_taken_and_right(checker, tmp_path, fmt, n, offsets, base):
    if fmt == "sym" and not any(o >= 0 for o in offsets):
        offsets = [-o for o in offsets]
    A = banded(n, offsets, n)
    x = np.random.default_rng(1).uniform(-1, 1, n)
    word, y = run(checker, tmp_path, fmt, arrays_of(A, fmt), x, base)
    if fmt == "sym" and offsets in ([3], [-3]):  # no diagonal entries: half of the positions are padding
        assert word == "NODIAGONALS"
        return
    assert word == "OK"
    same(y, *reference(A, x, fmt))


@pytest.mark.parametrize("fmt", ["csr", "sym", "csc"])
def test_holes_zeros_and_non_finite_elements(checker, tmp_path, fmt):
    # an absent entry adds nothing to its row even where x is inf or NaN; a stored zero does
    n = 500
    A = banded(n, [-20, -1, 0, 1, 20], 7, holes=0.2)
    A.data[::11] = 0.0
    A.data[5::11] = -0.0
    x = np.random.default_rng(2).uniform(-1, 1, n)
    x[[3, 77, 300]] = np.inf, -np.inf, np.nan
    arrays = arrays_of(A, fmt)
    word, y = run(checker, tmp_path, fmt, arrays, x)
    assert word == "OK"
    if fmt == "sym":
        U = sp.csr_matrix((arrays[2], arrays[1], arrays[0]), shape=(n, n))
        ref, scale = reference(U, x, "csr")
        L = sp.triu(U, 1).T.tocsr()
        r2, s2 = reference(L, x, "csr")
        with np.errstate(invalid="ignore"):
            ref, scale = ref + r2, scale + s2
    else:
        ref, scale = reference(A, x, fmt)
    same(y, ref, scale)


def test_turned_down(checker, tmp_path):
    rng = np.random.default_rng(3)
    for A in (banded(300, list(range(-16, 17)), 1),                    # 33 diagonals
              banded(300, [-7, -1, 0, 1, 7], 2, holes=0.5),            # half of the positions empty
              sp.random(400, 400, 0.02, random_state=4, format="csr") + sp.eye(400, format="csr")):
        A = A.tocsr()
        A.sort_indices()
        word, _ = run(checker, tmp_path, "csr", arrays_of(A, "csr"), rng.uniform(-1, 1, A.shape[0]))
        assert word == "NODIAGONALS"
    empty = (np.zeros(6, np.int32), np.zeros(0, np.int32), np.zeros(0))
    assert run(checker, tmp_path, "csr", empty, np.ones(5))[0] == "NODIAGONALS"


@pytest.mark.parametrize("grid", [(5, 5, 5), (9, 10, 11), (4, 30, 12)])
@pytest.mark.parametrize("fmt", ["csr", "sym", "csc"])
def test_finite_element_grids(checker, tmp_path, grid, fmt):
    s = femgen.build_system(femgen.Grid(*grid))
    arrays = {"csr": (s.ptr, s.idx, s.val), "sym": s.upper(), "csc": s.csc()}[fmt]
    x = femgen.random_vector(s.n, 4)
    word, y = run(checker, tmp_path, fmt, arrays, x)
    stored, K = arrays[1].shape[0], 8 if fmt == "sym" else 15
    assert word == ("OK" if 3 * stored >= 2 * K * s.n else "NODIAGONALS")
    if word == "OK":
        A = sp.csr_matrix((s.val, s.idx, s.ptr), shape=(s.n, s.n))
        same(y, *reference(A, x, "csr"))
