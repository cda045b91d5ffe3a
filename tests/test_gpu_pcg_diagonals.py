"""Single-reduction CG on the diagonal layout: ranges of one row per CTA up to
several rows per thread, idle CTAs, ragged ends and non-symmetric offsets,
against the same matrix's row-gather solve (not its iteration count: at 1e-12
one restart more or less from the drifted recurrences changes it by a third); and its time per iteration at the
published system size, where the one pass over the rows is what the variant is
for."""
import numpy as np
import pytest

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


def both(arrays, fmt, monkeypatch):
    D = gb.Matrix(fmt, *arrays)
    monkeypatch.setenv("GBCG_DIAGONALS", "0")
    O = gb.Matrix(fmt, *arrays)
    monkeypatch.delenv("GBCG_DIAGONALS")
    return D, O


@pytest.mark.parametrize("grid,ctas", [((4, 4, 5), None), ((12, 12, 12), None), ((17, 15, 19), "5"), ((12, 12, 12), "1"),
                                       ((31, 31, 32), None), ((31, 31, 32), "9"), ((9, 8, 7), "152")])
@pytest.mark.parametrize("fmt", ["csr", "csc"])
def test_solves(torch, grid, ctas, fmt, monkeypatch):
    s = fem(*grid)
    if ctas:
        monkeypatch.setenv("GBCG_GRID", ctas)
    arrays = (s.ptr, s.idx, s.val) if fmt == "csr" else s.csc()
    b = torch.from_numpy(s.b).cuda()
    D, O = both(arrays, fmt, monkeypatch)
    with D, O:
        x, i = D.solve(b, tol=1e-12, maxit=10 * s.n, variant="pipelined")
        z, j = O.solve(b, tol=1e-12, maxit=10 * s.n, variant="pipelined")
        again, _ = D.solve(b, tol=1e-12, maxit=10 * s.n, variant="pipelined")
    assert i.status == j.status == "OK" and torch.equal(x, again)
    r = s.b - oracle.spmv("csr", s.ptr, s.idx, s.val, x.cpu().numpy())
    assert np.linalg.norm(r) <= 1e-12 * np.linalg.norm(s.b)
    assert torch.linalg.norm(x - z) <= 1e-8 * torch.linalg.norm(z)


def test_iterations_are_not_slower_than_by_rows(torch, monkeypatch):
    s = femgen.build_system(femgen.PAPER_SIZE)
    b = torch.from_numpy(s.b).cuda()
    D, O = both((s.ptr, s.idx, s.val), "csr", monkeypatch)
    times = {D: [], O: []}
    with D, O:
        for _ in range(6):
            for M in (D, O):
                _, info = M.solve(b, tol=1e-10, maxit=10 * s.n, variant="pipelined")
                times[M].append(info.kernel_ms / info.iterations)
    assert min(times[D]) <= min(times[O]), times
