"""k_assemble on a pointer array that decreases: such a position has no
contributions, as a loop over [tptr[p], tptr[p + 1]) has it, and the others
are summed as they stand."""
import numpy as np
import pytest

import paper_1010_4639_gb300 as gb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count,lengths", [(3, 4), (255, 9), (600, 40), (1025, 3)])
def test_decreasing_pointers_are_empty_positions(count, lengths):
    import torch
    gb.build()
    rng = np.random.default_rng(count)
    tptr = np.concatenate([[0], np.cumsum(rng.integers(0, lengths, count))]).astype(np.int64)
    dips = np.arange(1, count, 3)
    tptr[dips] = np.maximum(0, tptr[dips - 1] - rng.integers(1, 60, dips.size))  # within the block's own range
    tptr[::256] = np.maximum.accumulate(tptr)[::256]  # a block of positions starts and ends in order
    tptr[-1] = tptr.max()
    nnz = int(tptr.max())
    telem = rng.integers(0, 50, nnz).astype(np.int32)
    tw, coef = rng.uniform(-1, 1, nnz), rng.uniform(0.5, 2.0, 50)
    tptr[dips] = np.maximum(tptr[dips], tptr[dips // 256 * 256])  # not before the block's first contribution
    out = gb.assemble(*(torch.from_numpy(a).cuda() for a in (tptr, telem, tw, coef))).cpu().numpy()
    for p in range(count):
        a, z = tptr[p], tptr[p + 1]
        ref = float(np.dot(tw[a:z], coef[telem[a:z]])) if z > a else 0.0
        assert abs(out[p] - ref) <= 1e-15 * max(1, z - a) * np.abs(tw[a:z]).sum() * 2.0 + 0.0
