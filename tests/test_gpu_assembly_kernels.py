"""The staged assembly kernels at the sizes where they can go wrong: counts
around a block's positions and elements, contributions around one stage,
positions without any, elements without any position, every pair count."""
import numpy as np
import pytest

import oracle
import paper_1010_4639_gb300 as gb

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -52


@pytest.fixture(scope="module")
def torch():
    import torch
    gb.build()
    assert torch.cuda.is_available()
    return torch


@pytest.mark.parametrize("nnz,longest", [(1, 1), (255, 3), (256, 1), (257, 40), (1000, 8), (300, 9000), (70000, 24)])
def test_assemble(torch, nnz, longest):
    rng = np.random.default_rng(nnz + longest)
    count = rng.integers(0, min(longest, 24) + 1, nnz)  # some positions have none
    count[::97] = longest  # also longer than a stage
    tptr = np.concatenate([[0], np.cumsum(count)]).astype(np.int64)
    ne = 500
    telem = rng.integers(0, ne, int(tptr[-1])).astype(np.int32)
    tw, coef = rng.uniform(-1, 1, int(tptr[-1])), rng.uniform(-1, 1, ne)
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    val = gb.assemble(T(tptr), T(telem), T(tw), T(coef)).cpu().numpy()
    # the kernel sums in the oracle's order; fused multiply-adds round once per term
    bound = np.array([np.abs(tw[a:b] * coef[telem[a:b]]).sum() for a, b in zip(tptr[:-1], tptr[1:])])
    assert np.all(np.abs(val - oracle.assemble(tptr, telem, tw, coef)) <= (count + 1) * EPS * bound)


@pytest.mark.parametrize("m", [0, 1, 2, 10, 15, 16, 17, 63, 64])
@pytest.mark.parametrize("ne", [1, 31, 257, 5000])
def test_element_grad(torch, ne, m):
    rng = np.random.default_rng(ne * 100 + m)
    nnz = 700
    pos = rng.integers(-1, nnz, (ne, m)).astype(np.int32)
    w, g = rng.uniform(-1, 1, (ne, m)), rng.uniform(-1, 1, nnz)
    pos[ne // 2] = -1
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    gc = gb.element_grad(T(pos), T(w), T(g)).cpu().numpy()
    terms = w * np.where(pos >= 0, g[np.maximum(pos, 0)], 0.0)
    assert np.all(np.abs(gc - terms.sum(axis=1)) <= (m + 2) * EPS * np.abs(terms).sum(axis=1))
    assert gc[ne // 2] == 0.0
