"""Cases that stand for what a program does with this library, for timing.

A case is a dict of plain values.  ``prepare`` builds what the program holds
before the call (matrix handle, vectors on the GPU), ``run`` makes the call
through the public entry points and returns its whole outputs, ``work`` gives
the bytes and operations one pass cannot do without, and ``exact`` the same
outputs from numpy in 64 bits.

Kinds of work:

* ``product``: y = A x, the call an outer iteration of the caller's own makes
  (an eigensolver, a time stepper, a residual check);
* ``solve``: conjugate gradient from x = 0 to a relative residual, in double
  precision, as single-precision iterations with double-precision updates, or
  as restarted refinement;
* ``batch``: many uneven systems with several right-hand sides each in one
  launch;
* ``differentiate``: coefficients -> stored values -> solution -> loss, forward
  and backward;
* ``assembly``: one step of a nonlinear or transient simulation without its
  solve: new coefficients -> stored values -> handle -> residual product, and
  the gradient kernels on the way back.

The systems are the seeded finite-element matrices of ``femgen``.  ``order``
is the numbering of the unknowns: "grid" keeps the generator's natural order,
"mesh" renumbers them at random within windows of consecutive unknowns, as an
unstructured mesh after a bandwidth reduction looks to the product.

Solves stop at tolerances at which the solution itself is determined (its
error stays below 1e-9 at these contrasts): with the default 1e-10 on a
contrast of 1000 two correct solves differ by more than their own rounding.
"""
import math

import numpy as np
import torch

import femgen
import paper_1010_4639_gb300 as gb

WINDOW = 2048  # unknowns of one renumbering window ("mesh" order)
RHS = 8


def _case(kind, dims, **options):
    nx, ny, nz = dims
    return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, **options}


def listed():
    cases = [
        # the smallest call: 1000 unknowns, all launch and latency
        ("product csr f64 smallest", _case("product", (12, 12, 12), fmt="csr", dtype="float64", order="grid")),
        # the published system size (31 x 31 x 32 nodes), symmetric storage, single precision
        ("product sym f32 paper size", _case("product", (31, 31, 32), fmt="sym", dtype="float32", order="grid")),
        # unstructured numbering, columns handed over (CSC), odd edges
        ("product csc f64 mesh order", _case("product", (61, 45, 53), fmt="csc", dtype="float64", order="mesh")),
        # a medium system in the symmetric storage FEM codes hold, double precision
        ("product sym f64 medium", _case("product", (96, 81, 90), fmt="sym", dtype="float64", order="grid")),
        # larger than any cache: 5 million unknowns, 73 million entries, single precision
        ("product csr f32 largest", _case("product", (192, 177, 154), fmt="csr", dtype="float32", order="grid")),
        # the published system solved as published: double precision throughout, latency-bound
        ("solve csr fp64 paper size",
         _case("solve", (31, 31, 32), fmt="csr", precision="fp64", order="grid", contrast=100.0, tol=1e-13)),
        # the benchmark's method on its 128^3 system: symmetric storage, reliable updates
        ("solve sym fp32_ru 128^3",
         _case("solve", (128, 128, 128), fmt="sym", precision="fp32_ru", order="grid", contrast=10.0, tol=1e-12)),
        # the same method on an unstructured numbering
        ("solve csr fp32_ru mesh order",
         _case("solve", (47, 39, 53), fmt="csr", precision="fp32_ru", order="mesh", contrast=10.0, tol=1e-12)),
        # restarted refinement (single-precision inner solves steered from the host)
        ("solve csr fp32_ir 96^3",
         _case("solve", (96, 96, 96), fmt="csr", precision="fp32_ir", order="grid", contrast=10.0, tol=1e-12)),
        # uneven systems with eight right-hand sides each, one launch, autotuned
        ("batch fp32_ru 48 systems",
         _case("batch", (12, 40, 0), count=48, precision="fp32_ru", contrast=100.0, tol=1e-13, mix=3)),
        # the 64^3 differentiable solve: double-precision forward and adjoint, coefficient gradients
        ("differentiate sym 64^3", _case("differentiate", (64, 64, 64), fmt="sym", contrast=10.0, tol=1e-12)),
        # a simulation step around the solve at the same size, full storage
        ("assembly csr 64^3", _case("assembly", (64, 64, 64), fmt="csr", contrast=10.0)),
    ]
    return [dict(c, name=name) for name, c in cases]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _dims(rng, lo, hi, rows):
    """Three edges in [lo, hi], spread over their logarithm, of at most ``rows`` nodes."""
    while True:
        d = tuple(_log_int(rng, lo, hi) for _ in range(3))
        if d[0] * d[1] * d[2] <= rows:
            return d


def draw(rng):
    kind = rng.choices(["product", "solve", "batch", "differentiate", "assembly"], [8, 7, 2, 2, 2])[0]
    fmt = rng.choice(["csr", "sym", "csc"])
    order = rng.choices(["grid", "mesh"], [3, 1])[0]
    if kind == "product":
        rows = 200_000 if order == "mesh" else 700_000 if fmt == "sym" else 4_000_000
        return _case(kind, _dims(rng, 6, 200, rows), fmt=fmt, dtype=rng.choice(["float64", "float32"]), order=order)
    if kind == "solve":
        rows = 120_000 if order == "mesh" else 500_000
        return _case(kind, _dims(rng, 8, 96, rows), fmt=fmt, precision=rng.choice(["fp64", "fp32_ru", "fp32_ir"]),
                     order=order, contrast=float(round(10 ** rng.uniform(0.0, 1.3), 2)), tol=1e-12)
    if kind == "batch":
        lo = _log_int(rng, 6, 14)
        return _case(kind, (lo, rng.randint(lo + 4, 34), 0), count=_log_int(rng, 4, 40),
                     precision=rng.choice(["fp32_ru", "fp32_ir", "fp64"]), contrast=30.0, tol=1e-13,
                     mix=rng.randint(0, 1 << 20))
    if kind == "differentiate":
        return _case(kind, _dims(rng, 8, 64, 150_000), fmt=fmt, contrast=float(round(10 ** rng.uniform(0.0, 1.0), 2)),
                     tol=1e-12)
    return _case(kind, _dims(rng, 8, 80, 250_000), fmt=fmt, contrast=10.0)


# ------------------------------------------------------------------ inputs
def _grid(case, seed, dims=None, contrast=None):
    nx, ny, nz = dims or (case["nx"], case["ny"], case["nz"])
    # 0.15 of the spacing: at 0.2 a large mesh can hold an inverted element
    return femgen.Grid(nx, ny, nz, contrast=contrast or case.get("contrast", 10.0), jitter=0.15, seed_mesh=seed,
                       seed_x=seed + 1)


def _renumber(n, ptr, idx, val, seed):
    """The matrix with its unknowns renumbered at random within windows."""
    rng = np.random.default_rng([seed, 17])
    old = np.argsort(np.arange(n) // WINDOW + rng.random(n) * 0.999, kind="stable")  # new -> old
    new = np.empty(n, dtype=np.int64)
    new[old] = np.arange(n)
    rows = np.repeat(new, np.diff(ptr))
    cols = new[idx]
    at = np.argsort(rows * n + cols, kind="stable")
    count = np.bincount(rows, minlength=n)
    return np.concatenate([[0], np.cumsum(count)]).astype(np.int32), cols[at].astype(np.int32), val[at]


def _full(case, seed):
    """The system's full CSR arrays (ptr, idx, val), exactly symmetric."""
    s = femgen.build_system(_grid(case, seed))
    if case.get("order") == "mesh":
        return _renumber(s.n, s.ptr, s.idx, s.val, seed)
    return s.ptr, s.idx, s.val


def _stored(fmt, full):
    """What the caller hands over: the upper triangle for "sym", all entries
    otherwise (the CSC arrays of a symmetric matrix are its CSR arrays)."""
    if fmt != "sym":
        return full
    ptr, idx, val = full
    return femgen.upper(ptr.shape[0] - 1, ptr, idx, val)


def _vector(n, seed, k=0):
    return np.random.default_rng([seed, k]).uniform(-1.0, 1.0, n)


def _multiply(ptr, idx, val, x):
    """A x of full CSR arrays in 64 bits (every row holds its diagonal)."""
    return np.add.reduceat(val * x[idx], ptr[:-1].astype(np.int64))


def _batch(case, seed):
    """Grids fixed by the case; meshes, coefficients' boxes and right-hand sides by the seed."""
    rng = np.random.default_rng(case["mix"])
    ptrs, idxs, vals, off, rows, xs, bs = [np.zeros(1, np.int64)], [], [], 0, [0], [], []
    for i in range(case["count"]):
        dims = tuple(int(v) for v in rng.integers(case["nx"], case["ny"] + 1, 3))
        contrast = float(10 ** rng.uniform(1.0, math.log10(case["contrast"])))
        s = femgen.build_system(_grid(case, seed * 64 + i, dims, contrast))
        x = _vector(s.n * RHS, seed, i).reshape(s.n, RHS)
        b = np.stack([_multiply(s.ptr, s.idx, s.val, x[:, k]) for k in range(RHS)], axis=1)
        ptrs.append(s.ptr[1:].astype(np.int64) + off)
        idxs.append(s.idx.astype(np.int64) + rows[-1])
        vals.append(s.val)
        off += s.nnz
        rows.append(rows[-1] + s.n)
        xs.append(x)
        bs.append(b)
    return (np.array(rows, np.int64), np.concatenate(ptrs).astype(np.int32), np.concatenate(idxs).astype(np.int32),
            np.concatenate(vals), np.concatenate(xs), np.concatenate(bs))


def _elements(case, seed, stored):
    """The mesh's elements and their map into the stored values."""
    el = femgen.elements(_grid(case, seed))
    pos, w = femgen.element_map(el, stored[0], stored[1], "sym" if case["fmt"] == "sym" else "csr")
    return el, pos, w


def _coefficients(case, seed, count):
    return np.random.default_rng([seed, 5]).uniform(0.5, case["contrast"], count)


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        row_off, ptr, idx, val, _, b = _batch(case, seed)
        return {"case": case, "batch": gb.Batch(row_off, ptr, idx, val, nrhs=RHS), "b": _gpu(b)}
    full = _full(case, seed)
    n = full[0].shape[0] - 1
    stored = _stored(case["fmt"], full)
    state = {"case": case}
    if kind == "product":
        state["A"] = gb.Matrix(case["fmt"], *stored)
        state["x"] = _gpu(_vector(n, seed).astype(case["dtype"]))
    elif kind == "solve":
        state["A"] = gb.Matrix(case["fmt"], *stored)
        state["b"] = _gpu(_multiply(*full, _vector(n, seed)))
    else:
        el, pos, w = _elements(case, seed, stored)
        tptr, telem, tw = femgen.assembly_map(pos, w, stored[1].shape[0])
        if kind == "differentiate":
            state["assemble"] = gb.Assembly(pos, w, tptr, telem, tw)
            state["solve"] = gb.SparseSolve(case["fmt"], *stored, tol=case["tol"])
            state["coef"] = _gpu(el.coef).requires_grad_()
            state["b"] = _gpu(_multiply(*full, _vector(n, seed))).requires_grad_()
            state["weight"] = _gpu(_multiply(*full, _vector(n, seed, 1)))  # loss = weight . x
        else:
            state["A"] = gb.Matrix(case["fmt"], *stored)
            state["pos"], state["w"] = _gpu(pos), _gpu(w)
            state["tptr"], state["telem"], state["tw"] = _gpu(tptr), _gpu(telem), _gpu(tw)
            state["ptr"], state["idx"] = _gpu(stored[0]), _gpu(stored[1])
            state["coef"] = _gpu(_coefficients(case, seed, el.count))
            state["x"], state["lam"] = _gpu(_vector(n, seed)), _gpu(_vector(n, seed, 1))
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "product":
        A, x = state["A"], state["x"]
        return A.spmv(x) if case["dtype"] == "float64" else A.spmv_f32(x)
    if kind == "solve":
        x, _ = state["A"].solve(state["b"], tol=case["tol"], maxit=100_000, precision=case["precision"])
        return x
    if kind == "batch":
        x, _, _ = state["batch"].solve(state["b"], tol=case["tol"], maxit=100_000, precision=case["precision"])
        return x
    if kind == "differentiate":
        x = state["solve"](state["assemble"](state["coef"]), state["b"])
        loss = torch.dot(state["weight"], x)
        gcoef, gb_ = torch.autograd.grad(loss, (state["coef"], state["b"]))
        return {"x": x.detach(), "coef_grad": gcoef, "b_grad": gb_}
    values = gb.assemble(state["tptr"], state["telem"], state["tw"], state["coef"])
    state["A"].update_values(values)
    y = state["A"].spmv(state["x"])
    grad = gb.grad_values(case["fmt"], state["ptr"], state["idx"], state["lam"], state["x"])
    coef_grad = gb.element_grad(state["pos"], state["w"], grad)
    return {"values": values, "y": y, "grad": grad, "coef_grad": coef_grad}


# ------------------------------------------------------- work and reference
def _sizes(nx, ny, nz):
    """(unknowns, entries of the full matrix, elements) of a grid whose faces are eliminated."""
    m = (nx - 2, ny - 2, nz - 2)
    n = m[0] * m[1] * m[2]
    off = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, 0, 1), (0, 1, 1), (1, 1, 1)]
    pairs = sum(math.prod(max(0, e - o) for e, o in zip(m, d)) for d in off)
    return n, n + 2 * pairs, 6 * (nx - 1) * (ny - 1) * (nz - 1)


def _iterations(edge, contrast, tol):
    """Iterations of a solve, from runs on this generator's systems: they grow
    with the edge, the square root of the condition number and the digits."""
    return 1.2 * edge * max(1.0, contrast) ** 0.42 / 2.63 * -math.log10(tol)


def work(case):
    """Each input read once and each output written once (4-byte indices; the
    matrix as handed over), and the multiply-adds of the products and vector
    updates: for a solve those of its iterations."""
    kind = case["kind"]
    if kind == "batch":
        rng = np.random.default_rng(case["mix"])
        nbytes = flops = 0.0
        for _ in range(case["count"]):
            dims = [int(v) for v in rng.integers(case["nx"], case["ny"] + 1, 3)]
            contrast = float(10 ** rng.uniform(1.0, math.log10(case["contrast"])))
            n, nnz, _ = _sizes(*dims)
            nbytes += 12 * nnz + 4 * n + 16 * n * RHS
            flops += _iterations(max(dims), contrast, case["tol"]) * RHS * (2 * nnz + 10 * n)
        return {"bytes": nbytes, "flops": flops}
    n, nnz, elements = _sizes(case["nx"], case["ny"], case["nz"])
    stored = (nnz + n) // 2 if case["fmt"] == "sym" else nnz
    edge = max(case["nx"], case["ny"], case["nz"])
    if kind == "product":
        v = 8 if case["dtype"] == "float64" else 4
        return {"bytes": (v + 4) * stored + 4 * n + 2 * v * n, "flops": 2 * nnz}
    if kind == "solve":
        iterations = _iterations(edge, case["contrast"], case["tol"])
        return {"bytes": 12 * stored + 4 * n + 16 * n, "flops": iterations * (2 * nnz + 10 * n)}
    pairs = 10 if case["fmt"] == "sym" else 16
    maps = 12 * pairs * elements + 16 * elements  # the element map read once, coefficients in, gradients out
    if kind == "differentiate":
        iterations = 2 * _iterations(edge, case["contrast"], case["tol"])
        return {"bytes": 2 * maps + 4 * stored + 32 * n, "flops": iterations * (2 * nnz + 10 * n)}
    return {"bytes": 2 * maps + 12 * stored + 8 * stored + 8 * stored + 40 * n,
            "flops": 2 * nnz + 4 * pairs * elements + 3 * stored}


def _gradient(fmt, stored, lam, x):
    """dL/d(stored values) of L(x), A x = b, for the adjoint lam."""
    ptr, idx, _ = stored
    rows = np.repeat(np.arange(ptr.shape[0] - 1), np.diff(ptr))
    if fmt == "csc":
        return -lam[idx] * x[rows]
    if fmt == "csr":
        return -lam[rows] * x[idx]
    return np.where(rows == idx, -lam[rows] * x[idx], -(lam[rows] * x[idx] + lam[idx] * x[rows]))


def _element_gradient(el, lam, x):
    """dL/dcoef per element: -lam' Kh x over its unknowns."""
    l4 = np.where(el.nodes >= 0, lam[el.nodes], 0.0)
    x4 = np.where(el.nodes >= 0, x[el.nodes], 0.0)
    return -np.einsum("ea,eab,eb->e", l4, el.kh, x4)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return torch.from_numpy(_batch(case, seed)[4])
    full = _full(case, seed)
    n = full[0].shape[0] - 1
    if kind == "product":
        return torch.from_numpy(_multiply(*full, _vector(n, seed).astype(case["dtype"]).astype(np.float64)))
    x, lam = _vector(n, seed), _vector(n, seed, 1)
    if kind == "solve":
        return torch.from_numpy(x)
    stored = _stored(case["fmt"], full)
    el, pos, w = _elements(case, seed, stored)
    if kind == "differentiate":
        return {"x": torch.from_numpy(x), "coef_grad": torch.from_numpy(_element_gradient(el, lam, x)),
                "b_grad": torch.from_numpy(lam)}
    coef = _coefficients(case, seed, el.count)
    values = np.zeros(stored[1].shape[0])
    for k in range(pos.shape[1]):
        there = pos[:, k] >= 0
        values += np.bincount(pos[there, k], weights=(coef * w[:, k])[there], minlength=values.shape[0])
    ptr, idx = stored[0], stored[1]
    rows = np.repeat(np.arange(n), np.diff(ptr))
    if case["fmt"] == "csc":
        rows, cols = idx, rows
    else:
        cols = idx
    y = np.bincount(rows, weights=values * x[cols], minlength=n)
    if case["fmt"] == "sym":
        off = rows != cols
        y += np.bincount(cols[off], weights=(values * x[rows])[off], minlength=n)
    grad = _gradient(case["fmt"], stored, lam, x)
    return {"values": torch.from_numpy(values), "y": torch.from_numpy(y), "grad": torch.from_numpy(grad),
            "coef_grad": torch.from_numpy(_element_gradient(el, lam, x))}
