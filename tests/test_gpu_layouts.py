"""The tests of products, solves, asynchronous solves and updates once more on
the layouts that a matrix numbered line by line no longer takes by itself: rows
(16- and 32-bit columns) for full storage and tiles for symmetric storage.
Each test states the layouts its handles ran on."""
import itertools

import pytest

import paper_1010_4639_gb300 as gb
import test_gpu_async
import test_gpu_cg
import test_gpu_golden
import test_gpu_grad
import test_gpu_pcg
import test_gpu_ru
import test_gpu_spmv
import femgen

pytestmark = pytest.mark.gpu
ROWS, PLAN, TILES = 0, 1, 2


@pytest.fixture(scope="module")
def torch():
    import torch
    gb.build()
    assert torch.cuda.is_available()
    return torch


@pytest.fixture(scope="module")
def s128():
    return femgen.build_system(femgen.LARGE)


@pytest.fixture
def products(monkeypatch):
    """No diagonals; the layouts of the handles made meanwhile."""
    seen = set()

    class Seen(gb.Matrix):
        def __init__(self, *args, **kwargs):
            super().__init__(*args, **kwargs)
            if self.n:
                seen.add(self.stats()["product"])

    monkeypatch.setenv("GBCG_DIAGONALS", "0")
    monkeypatch.setattr(gb, "Matrix", Seen)
    return seen


def cases(test, keep=lambda kw: True):
    """The test's parameter sets, from its own marks."""
    sets = [[dict(zip(m.args[0].split(","), v if "," in m.args[0] else (v,))) for v in m.args[1]]
            for m in getattr(test, "pytestmark", []) if m.name == "parametrize"]
    out = [dict(itertools.chain.from_iterable(d.items() for d in s)) for s in itertools.product(*sets)]
    return [pytest.param(test, kw, id=f"{test.__name__}-" + "-".join(str(v).replace(" ", "") for v in kw.values()))
            for kw in out if keep(kw)]


def full(kw):
    return kw.get("fmt", "csr") in ("csr", "csc")


def run(test, kw, torch, monkeypatch, products, s128):
    given = {"torch": torch, "monkeypatch": monkeypatch, "s128": s128}
    names = test.__code__.co_varnames[:test.__code__.co_argcount]
    test(**{k: given[k] for k in names if k in given}, **kw)
    return products


@pytest.mark.parametrize("test,kw", cases(test_gpu_spmv.test_fem_spmv_matches_oracle, full)
                         + cases(test_gpu_spmv.test_fp32_product, full)
                         + cases(test_gpu_spmv.test_narrow_and_wide_indices_agree)
                         + cases(test_gpu_spmv.test_one_shot_product_many_slices_per_warp)
                         + cases(test_gpu_cg.test_fp64_cg_matches_oracle, full)
                         + cases(test_gpu_cg.test_mixed_precision_refinement, full)
                         + cases(test_gpu_ru.test_reliable_updates_match_oracle, full)
                         + cases(test_gpu_ru.test_reliable_updates_edge_cases)
                         + cases(test_gpu_pcg.test_pipelined_matches_oracle, full)
                         + cases(test_gpu_pcg.test_pipelined_edge_cases)
                         + cases(test_gpu_pcg.test_pipelined_grid_sizes)
                         + cases(test_gpu_pcg.test_pipelined_full_size)
                         + cases(test_gpu_async.test_async_equals_sync, full)
                         + cases(test_gpu_async.test_async_statuses)
                         + cases(test_gpu_async.test_async_solve_in_a_cuda_graph)
                         + cases(test_gpu_grad.test_update_values_equals_a_fresh_handle, full)
                         + cases(test_gpu_golden.test_128_fp64, full)
                         + cases(test_gpu_golden.test_128_reliable_updates, full))
def test_rows(test, kw, torch, monkeypatch, products, s128):
    assert ROWS in run(test, kw, torch, monkeypatch, products, s128) and not products & {3, 4}


def tiles(kw):
    return kw.get("fmt") in ("sym", "tiles")


@pytest.mark.parametrize("test,kw", cases(test_gpu_spmv.test_fem_spmv_matches_oracle, tiles)
                         + cases(test_gpu_spmv.test_fp32_product, tiles)
                         + cases(test_gpu_cg.test_fp64_cg_matches_oracle, tiles)
                         + cases(test_gpu_cg.test_mixed_precision_refinement, tiles)
                         + cases(test_gpu_cg.test_host_memory_path_and_determinism)
                         + cases(test_gpu_ru.test_reliable_updates_match_oracle, lambda kw: kw["fmt"] == "tiles")
                         + cases(test_gpu_ru.test_reliable_updates_tiled_layout_edge_cases)
                         + cases(test_gpu_ru.test_reliable_updates_tiled_layout_grid_sizes)
                         + cases(test_gpu_ru.test_streamed_vector_passes)
                         + cases(test_gpu_pcg.test_pipelined_rejects_the_tiled_layout)
                         + cases(test_gpu_async.test_async_equals_sync, tiles)
                         + cases(test_gpu_grad.test_update_values_equals_a_fresh_handle, tiles)
                         + cases(test_gpu_golden.test_128_fp64, tiles)
                         + cases(test_gpu_golden.test_128_reliable_updates, tiles)
                         + cases(test_gpu_golden.test_128_restarted_refinement))
def test_tiles(test, kw, torch, monkeypatch, products, s128):
    assert run(test, kw, torch, monkeypatch, products, s128) == {TILES}


def test_full_size_products(torch, monkeypatch, products, s128):
    run(test_gpu_spmv.test_full_size_128_all_formats, {}, torch, monkeypatch, products, s128)
    assert products == {ROWS, TILES}


@pytest.mark.parametrize("ctas", ["1", "7", "64"])
def test_grid_sizes(torch, ctas, monkeypatch, products, s128):
    run(test_gpu_cg.test_grid_sizes, {"grid_ctas": ctas}, torch, monkeypatch, products, s128)
    assert products and not products & {3, 4}


@pytest.mark.parametrize("wide", ["0", "1"])
def test_single_reduction_on_scattered_rows(torch, wide, monkeypatch, products):
    # long rows, empty slices' ends, 16- and 32-bit columns
    import numpy as np

    import oracle
    from gpu_cases import random_spd
    monkeypatch.setenv("GBCG_WIDE_INDEX", wide)
    ptr, idx, val = random_spd(2999, 9, density=0.003, dense_rows=(7, 1500, 2998))
    b = np.random.default_rng(1).uniform(-1, 1, 2999)
    ref = oracle.cg("csr", ptr, idx, val, b, tol=1e-12)
    for fmt in ("csr", "csc"):  # a symmetric matrix: its columns are its rows
        with gb.Matrix(fmt, ptr, idx, val) as A:
            assert A.stats()["long_rows"] >= 1 and A.stats()["index_bytes"] == (4 if wide == "1" else 2)
            x, info = A.solve(torch.from_numpy(b).cuda(), tol=1e-12, variant="pipelined")
        assert info.status == "OK"
        assert np.linalg.norm(x.cpu().numpy() - ref.x) <= 1e-8 * np.linalg.norm(ref.x)
    assert products == {ROWS}
