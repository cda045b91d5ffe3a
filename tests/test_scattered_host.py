"""The row-gather layout of symmetric storage with scattered neighbours
(csrc/layout.cpp, build_sym_full) on the CPU: the full operator's row sums
against the upper triangle's, and when a slice fits a tile, over ragged sizes,
index bases, missing diagonals, stored zeros, empty and long rows."""
import os
import struct
import subprocess

import numpy as np
import pytest
import scipy.sparse as sp

import femgen

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1010_4639_gb300", "csrc")


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("scattered") / "scattered_check")
    subprocess.run(["g++", "-O1", "-std=c++17", os.path.join(HERE, "scattered_check.cpp"),
                    os.path.join(CSRC, "layout.cpp"), "-o", out], check=True)
    return out


def check(checker, tmp_path, U, base, slot_cap=2048, ent_cap=4096):
    n = U.shape[0]
    x = np.random.default_rng(n).uniform(-1, 1, n)
    src, dst = str(tmp_path / "m.bin"), str(tmp_path / "y.bin")
    with open(src, "wb") as f:
        f.write(struct.pack("<qq", n, U.nnz))
        for a, t in ((U.indptr + base, np.int32), (U.indices + base, np.int32), (U.data, np.float64), (x, np.float64)):
            f.write(np.ascontiguousarray(a, dtype=t).tobytes())
    out = subprocess.run([checker, src, str(base), str(slot_cap), str(ent_cap), dst], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
    ref = U @ x + sp.triu(U, 1).T @ x
    # two summation orders of at most m terms: 2 m eps of the terms' sizes, m below 1000 here
    scale = abs(U) @ abs(x) + abs(sp.triu(U, 1)).T @ abs(x)
    assert np.all(np.abs(np.fromfile(dst) - ref) <= 5e-13 * scale)
    word = out.stdout.split()
    return float(word[1]), bool(int(word[2]))


@pytest.mark.parametrize("base", [0, 1])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 200, 1025, 4097])
def test_random_upper_triangles(checker, tmp_path, n, base):
    U = sp.triu(sp.random(n, n, min(1.0, 6 / n), random_state=n, format="csr")).tocsr()
    U.data[::7] = 0.0
    if n >= 200:  # a long row, reached from both sides
        d = sp.lil_matrix((n, n))
        d[n // 2, :] = 1.5
        d[:, n // 2] = 1.5
        U = sp.triu(U + d.tocsr()).tocsr()
    U.sort_indices()
    check(checker, tmp_path, U, base)
    check(checker, tmp_path, U, base, slot_cap=256, ent_cap=512)


@pytest.mark.parametrize("grid", [(9, 10, 11), (17, 15, 19), (31, 31, 32)])
def test_numberings(checker, tmp_path, grid):
    s = femgen.build_system(femgen.Grid(*grid))
    A = sp.csr_matrix((s.val, s.idx, s.ptr), shape=(s.n, s.n))
    lines, _ = check(checker, tmp_path, sp.triu(A).tocsr(), 0)
    p = np.random.default_rng(1).permutation(s.n)
    U = sp.triu(A[p][:, p]).tocsr()
    U.sort_indices()
    mixed, fits = check(checker, tmp_path, U, 0)
    # a tile of a small matrix has few rows, which reach few windows in any numbering
    assert fits and lines <= 8 and (mixed > 16 if s.n > 4096 else mixed >= lines)
