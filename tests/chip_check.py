"""Compiles tests/chip_check.cu (inputs and entries of the scalar tests)."""
from __future__ import annotations

import ctypes
import os
import subprocess

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))


def load(folder):
    from paper_1010_4639_gb300 import builder
    out = os.path.join(str(folder), "chip_check.so")
    subprocess.run([builder._nvcc(), "-O2", "-std=c++17", *builder.ARCH, "-shared", "-Xcompiler", "-fPIC", "-I",
                    builder.INCLUDE, os.path.join(HERE, "chip_check.cu"), "-o", out], check=True)
    return ctypes.CDLL(out)


def addr(a):
    return ctypes.c_void_p(a.data_ptr() if hasattr(a, "data_ptr") else a.ctypes.data)


def dividends_and_divisors(n=1 << 20, seed=3):
    """Pairs over the whole range of double precision: random significands at
    random exponents, significands next to powers of two and to each other, exact and nearly
    exact quotients, and every special value against every other."""
    rng = np.random.default_rng(seed)
    bits = rng.integers(0, 1 << 63, (2, n), dtype=np.uint64)
    any_ = bits.view(np.float64)
    near = rng.uniform(1.0, 2.0, (2, n)) * 2.0 ** rng.integers(-60, 60, (2, n))
    edge = (np.array([0, 1, 2, 3, (1 << 52) - 1, (1 << 52) - 2, 1 << 51, (1 << 51) + 1, (1 << 24) - 1, 1 << 24],
                     np.uint64)[rng.integers(0, 10, (2, n // 4))] | np.uint64(1023 << 52)).view(np.float64)
    d = near[0][: n // 4]
    q = near[1][: n // 4]
    exact = np.stack([(d.astype(np.float32) * q.astype(np.float32).astype(np.float64)), d.astype(np.float32)])
    close = np.stack([np.nextafter(d * q, np.inf), d])
    special = np.array([0.0, -0.0, 5e-324, 2.2250738585072014e-308, 1e-300, 1.0, -1.0, 1.7976931348623157e308, np.inf,
                        -np.inf, np.nan, np.nextafter(1.0, 0.0), np.nextafter(1.0, 2.0)])
    pairs = np.stack([x.ravel() for x in np.meshgrid(special, special)])
    return np.ascontiguousarray(np.concatenate([any_, near, edge, exact, close, pairs], axis=1))


def same(a, b):
    """Equal bits, any NaN equal to any NaN."""
    return np.all((a.view(np.uint64) == b.view(np.uint64)) | (np.isnan(a) & np.isnan(b)))
