"""Compiles tests/chip_check.cu (inputs and entries of the scalar tests)."""
from __future__ import annotations

import ctypes
import os
import subprocess
from fractions import Fraction

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


def sums(G, seed=5):
    """(partial sums [cases, G], sums an iteration earlier [cases]): positive and mixed partial
    sums whose total lies 2^-20 .. 2^18 from the earlier sum, one that
    outweighs all others, zeros, the ends of the range, infinities and NaN."""
    rng = np.random.default_rng(seed)
    part, prev = [], []
    for scale in (1.0, 3e-150, 7e140, 1e-290, 1e290, 5e-324, 0.0, -2.0, np.inf, np.nan):
        for ratio in range(-20, 19):
            for kind in range(3):
                p = rng.uniform(0.0, 1.0, G)
                if kind == 1:
                    p[rng.random(G) < 0.5] *= -1.0
                    p[0] = 2.0 * G  # the total stays positive
                if kind == 2:
                    p = p * 2.0 ** -rng.integers(0, 90, G)
                    p[rng.integers(0, G)] = 1.0
                with np.errstate(over="ignore", invalid="ignore", under="ignore"):
                    base = scale if 1e-300 < scale < 1e300 else 1.0
                    part.append(p / p.sum() * rng.uniform(0.6, 1.4) * 2.0 ** ratio * base)
                prev.append(scale)
    for special in (0.0, -1.0, np.inf, -np.inf, np.nan, 2.0 ** 40):
        part.append(np.where(np.arange(G) == G // 2, special, 2.0 ** -30))
        prev.append(1.0)
    return np.array(part), np.array(prev)


def check_sum(part, prev, got, retaken):
    """The sum against the exact one.  A fixed-point sum is off by its
    truncations, a quarter of its last bit, and the conversion's roundings: one
    half (two where it exceeds 2^20 of the earlier sum).  A sum of doubles by
    at most one rounding of the partial sums' total size per addition."""
    if not np.all(np.isfinite(part)):
        assert retaken
        with np.errstate(invalid="ignore"):
            want = part.sum()
        assert np.isnan(got) if np.isnan(want) else got == want
        return
    total = sum(map(Fraction, part.tolist()))
    error, exact = abs(Fraction(float(got)) - total), float(total)
    if retaken:
        assert error <= len(part) * Fraction(2) ** -53 * sum(map(Fraction, np.abs(part).tolist()))
    else:
        ulps = 0.25 + (0.5 if exact < 2.0 ** 20 * prev else 1.0)
        assert error <= Fraction(ulps) * Fraction(float(np.spacing(exact))), (exact, prev)
    # taken again or not, by the sums' size
    if 1e-200 < prev < 1e200:
        if 2.0 ** -9 * prev <= exact and max(abs(part)) < 2.0 ** 14 * prev:
            assert not retaken
        if exact < 2.0 ** -11 * prev or max(abs(part)) >= 2.0 ** 16 * prev:
            assert retaken
