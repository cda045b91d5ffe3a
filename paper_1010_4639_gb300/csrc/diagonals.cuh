// diagonals.cuh -- device code of the diagonal layout (layout.h, DiaHost).
//
// A finite-element matrix on a mesh numbered line by line holds few distinct
// column offsets (15 for linear tetrahedra on a box).  Its values are stored
// by diagonal, val[k * ld + i] = A(i, i + off[k]), and no indices at all:
// every load of a warp is contiguous, and no load's address depends on
// another load.  The row-gather layout waits for the stage, then the columns,
// then the vector (about 3 100 cycles per 32 rows on GB300), and the
// symmetric tiles spend a CTA barrier per round.
//
// Symmetric storage keeps the diagonals off >= 0 only: A(i, i - off) is the
// value that row i - off holds, read again with an offset of its own (from L1
// or L2: HBM sees each value once).  Rows are summed in increasing column
// order, as the row-gather layout does, so full storage gives the same bits.
//
// Bound: HBM for the single-precision product, the FP64 pipe (two FMAs per
// cycle and SM) for the double-precision one.  What stood in the way was the
// instructions around the loads: one row per thread, with a bounds and a
// padding test per entry, kept 66% of the issue slots busy and took 29 us for
// the single-precision symmetric product at 128^3 (now 16; the tiles take 37).
// So a thread takes R rows
// 32 apart (one address per diagonal, the rows by immediate offsets), bounds
// are looked at once per segment, and padding is not tested at all: a
// position no entry was given for holds -0.0, which adds nothing unless x is
// not finite there, and a row whose sum is not finite is summed again entry by
// entry (0 * inf is not 0, and a stored zero is kept as +0.0).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "layout.h"

namespace gbcg {

template <typename V>
struct DiaDev {
  int64_t n = 0, ld = 0;
  const V* __restrict__ val = nullptr;
  int32_t K = 0;
  int32_t lo = 0, hi = 0;  // least and greatest column offset of the operator
  int32_t off[kMaxDiag] = {};
};

constexpr int kDiaThreads = 1024;  // persistent solvers: 32 warps of 64 registers
constexpr int kDiaBlock = 256;     // one-shot product

__device__ __forceinline__ bool dia_stored(float v) { return __float_as_uint(v) != 0x80000000u; }
__device__ __forceinline__ bool dia_stored(double v) {
  return (unsigned long long)__double_as_longlong(v) != 0x8000000000000000ull;
}
__device__ __forceinline__ bool dia_finite(float v) { return (__float_as_uint(v) & 0x7f800000u) != 0x7f800000u; }
__device__ __forceinline__ bool dia_finite(double v) {
  return ((unsigned)__double2hiint(v) & 0x7ff00000u) != 0x7ff00000u;
}
// Stored form of an entry's value (the padding marker is -0.0).
template <typename V>
__host__ __device__ __forceinline__ V dia_value(V v) { return v == V(0) ? V(0) : v; }

__device__ __forceinline__ double dia_fma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float dia_fma(float a, float b, float c) { return fmaf(a, b, c); }

template <bool NC, typename V>
__device__ __forceinline__ V dia_x(const V* x) {
  if constexpr (NC) return __ldg(x);
  else return *x;
}

// Where the loops below find a diagonal: the index of its first value and its
// column offset.  The one-shot kernels read their parameters; the persistent
// solvers a copy in shared memory, whose address fresh() hides from the
// compiler so that each half of each segment reads it again (kept in registers
// across the iteration, the diagonals' addresses spill: 2 KB per thread).
template <typename V>
struct DiaParam {
  const DiaDev<V>& A;
  __device__ __forceinline__ DiaParam fresh() const { return *this; }
  __device__ __forceinline__ int2 operator()(int k) const {
    return make_int2((int)((uint32_t)k * (uint32_t)A.ld), A.off[k]);
  }
};
struct DiaShared {
  uint32_t tab;
  __device__ __forceinline__ DiaShared fresh() const {
    DiaShared s = *this;
    asm volatile("" : "+r"(s.tab));
    return s;
  }
  __device__ __forceinline__ int2 operator()(int k) const {
    int2 d;
    asm("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(d.x), "=r"(d.y) : "r"(tab + 8 * k));
    return d;
  }
};
template <typename V>
struct alignas(16) DiaTab {
  int2 e[kMaxDiag];
  const V* val;
  int32_t n, K, lo, hi;
  __device__ __forceinline__ DiaShared entries() const {
    DiaShared s;
    s.tab = (uint32_t)__cvta_generic_to_shared(e);
    return s;
  }
};
// Every thread of the CTA calls it; a __syncthreads must follow.
template <typename V>
__device__ __forceinline__ void dia_tab_init(DiaTab<V>& t, const DiaDev<V>& A) {
  if (threadIdx.x < (unsigned)A.K)
    t.e[threadIdx.x] = make_int2((int)((uint32_t)threadIdx.x * (uint32_t)A.ld), A.off[threadIdx.x]);
  if (threadIdx.x == 0) {
    t.val = A.val;
    t.n = (int32_t)A.n;
    t.K = A.K;
    t.lo = A.lo;
    t.hi = A.hi;
  }
}

// Rows i, i + 32, ... (R of them): acc[r] gains the terms of half a row, in
// increasing column order -- MIRROR: columns i - off[k], k = K - 1 .. 1, whose
// values rows i - off[k] hold; else columns i + off[k], k = 0 .. K - 1.  The
// loads of C diagonals are issued before the first is used.  DESC: k from K - 1
// down.  CLAMP (segments
// at the ends of the matrix): rows past `last` are taken as `last`, columns
// outside the matrix as its first or last one; the value there is padding (a
// diagonal is stored with max(off) padding after its n values, where the
// mirrored index of the rows below off[k] leads).  A branch per diagonal
// around the clamps, or reading the CTA's own columns from shared memory, were
// both slower (25 000 -> 31 000 cycles per product at 128^3).
template <bool MIRROR, bool NC, bool CLAMP, bool DESC, int C, int R, typename V, class E>
__device__ __forceinline__ void dia_half(const E& table, int K, const V* val, int n, int last, int i0, const V* x,
                                         V (&acc)[R]) {
  const E entry = table.fresh();
  const int cnt = MIRROR ? K - 1 : K;
  for (int kb = 0; kb < cnt; kb += C) {
    V v[C][R], xv[C][R];
#pragma unroll
    for (int j = 0; j < C; ++j) {
      // past the last diagonal: the last one again, unused (no branches around the loads)
      const int m = min(kb + j, cnt - 1);
      const int2 d = entry(MIRROR || DESC ? K - 1 - m : m);
      if constexpr (!CLAMP) {
        const int c = MIRROR ? i0 - d.y : i0 + d.y;
        const V* pv = val + ((uint32_t)d.x + (uint32_t)(MIRROR ? c : i0));
        const V* px = x + c;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          v[j][r] = __ldg(pv + 32 * r);
          xv[j][r] = dia_x<NC>(px + 32 * r);
        }
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int i = min(i0 + 32 * r, last), c = MIRROR ? i - d.y : i + d.y;
          v[j][r] = __ldg(val + ((uint32_t)d.x + (uint32_t)(MIRROR ? c : i)));
          xv[j][r] = dia_x<NC>(x + min(max(c, 0), n - 1));
        }
      }
    }
#pragma unroll
    for (int j = 0; j < C; ++j)
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (kb + j < cnt) acc[r] = dia_fma(v[j][r], xv[j][r], acc[r]);
  }
}

template <bool SYM, typename V>
__host__ __device__ constexpr bool dia_apart() { return SYM && sizeof(V) == 4; }

// (A x)_i entry by entry: padding and columns outside the matrix are skipped.
template <bool SYM, bool NC, typename V, class E>
__device__ __forceinline__ V dia_row_exact(const E& table, int K, const V* val, int n, int i, const V* x) {
  const E entry = table.fresh();
  V acc = V(0), low = V(0);
  if constexpr (SYM)
#pragma unroll 1
    for (int k = K - 1; k > 0; --k) {
      const int2 d = entry(k);
      const int c = i - d.y;
      if (c < 0) continue;
      const V v = __ldg(val + ((uint32_t)d.x + (uint32_t)c));
      if (dia_stored(v)) low = dia_fma(v, dia_x<NC>(x + c), low);
    }
  if constexpr (!dia_apart<SYM, V>()) acc = low;
#pragma unroll 1
  for (int m = 0; m < K; ++m) {
    const int2 d = entry(dia_apart<SYM, V>() ? K - 1 - m : m);
    const int c = i + d.y;
    if (c < 0 || c >= n) continue;
    const V v = __ldg(val + ((uint32_t)d.x + (uint32_t)i));
    if (dia_stored(v)) acc = dia_fma(v, dia_x<NC>(x + c), acc);
  }
  return dia_apart<SYM, V>() ? low + acc : acc;
}

// acc[r] = (A x) of rows base + lane + 32 r up to `last` (base the warp's
// first row; what acc holds for rows past `last` is of no use).  HALO: x has
// kDiaHalo finite elements beyond max(off) on either side, so every column
// can be read; otherwise the segments at the ends of the matrix clamp (36 700
// cycles instead of 25 400 for the first and last CTA's product at 128^3, for
// which every other CTA then waits).
template <bool SYM, bool NC, bool HALO, int C, int R, typename V, class E>
__device__ __forceinline__ void dia_segment(const E& entry, int K, int lo, int hi, const V* val, int n, int last,
                                            int base, const V* x, V (&acc)[R]) {
  const int i0 = base + (threadIdx.x & 31);
#pragma unroll
  for (int r = 0; r < R; ++r) acc[r] = V(0);
  // single-precision symmetric rows sum the columns below and above the
  // diagonal apart and take the diagonal, the largest term, last, as the tiles
  // do: shorter and smaller sums round less (one sum: 8.1e-8 on a
  // finite-element matrix, the tiles 5.5e-8); double precision goes on with one sum, as full
  // storage does
  constexpr bool kApart = dia_apart<SYM, V>();
  V low[R];
#pragma unroll
  for (int r = 0; r < R; ++r) low[r] = V(0);
  if (HALO || (base + lo >= 0 && base + 32 * R - 1 + hi < n && base + 32 * R - 1 <= last)) {
    if constexpr (SYM) dia_half<true, NC, false, false, C, R>(entry, K, val, n, last, i0, x, kApart ? low : acc);
    dia_half<false, NC, false, kApart, C, R>(entry, K, val, n, last, i0, x, acc);
  } else {
    if constexpr (SYM) dia_half<true, NC, true, false, C, R>(entry, K, val, n, last, i0, x, kApart ? low : acc);
    dia_half<false, NC, true, kApart, C, R>(entry, K, val, n, last, i0, x, acc);
  }
  if constexpr (kApart)
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = low[r] + acc[r];
#pragma unroll
  for (int r = 0; r < R; ++r)
    if (!dia_finite(acc[r])) acc[r] = dia_row_exact<SYM, NC>(entry, K, val, n, min(i0 + 32 * r, last), x);
}

// Diagonals in flight, for K of them: chunks of eight would read one or two
// diagonals eight times over (2.0 M rows, symmetric, two stored diagonals,
// double precision: 58 us for a product in chunks of eight, 19 in chunks of two,
// tiles 41; three stored diagonals 58, 31 and 49).  Chosen once per product: at
// the end of every row's diagonals it cost the 15-diagonal products 1-3%.
__host__ __device__ constexpr int dia_few(int K) { return K <= 2 ? 2 : K <= 4 ? 4 : 8; }

// f(row, (A x)_row) for the rows [r0, r1) of the CTA.
template <bool SYM, bool HALO, int C, int R, typename V, class F>
__device__ __forceinline__ void dia_rows_in(const DiaTab<V>& t, int r0, int r1, const V* x, F&& f) {
  const int lane = threadIdx.x & 31, step = blockDim.x * R;
  for (int base = r0 + (threadIdx.x >> 5) * 32 * R; base < r1; base += step) {
    V acc[R];
    dia_segment<SYM, false, HALO, C, R>(t.entries(), t.K, t.lo, t.hi, t.val, t.n, r1 - 1, base, x, acc);
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (base + lane + 32 * r < r1) f(base + lane + 32 * r, acc[r]);
  }
}
template <bool SYM, bool HALO, int C, int R, typename V, class F>
__device__ __forceinline__ void dia_rows(const DiaTab<V>& t, int r0, int r1, const V* x, F&& f) {
  if constexpr (C == 8) {
    if (dia_few(t.K) == 2) return dia_rows_in<SYM, HALO, 2, R>(t, r0, r1, x, f);
    if (dia_few(t.K) == 4) return dia_rows_in<SYM, HALO, 4, R>(t, r0, r1, x, f);
  }
  dia_rows_in<SYM, HALO, C, R>(t, r0, r1, x, f);
}

// Product of the solvers whose vectors stay in global memory: rows per thread
// and diagonals in flight.
template <typename V>
__host__ __device__ constexpr int dia_r() { return sizeof(V) == 4 ? 4 : 1; }
template <typename V>
__host__ __device__ constexpr int dia_c() { return sizeof(V) == 4 ? 4 : 8; }

// y = A x on the rows [r0, r1) of the CTA.
template <typename V, bool SYM>
__device__ __forceinline__ void dia_product(const DiaTab<V>& t, int64_t r0, int64_t r1, const V* x, V* y) {
  dia_rows<SYM, false, dia_c<V>(), dia_r<V>()>(t, (int)r0, (int)r1, x, [&](int i, V q) { y[i] = q; });
}

// y = A x over the whole grid's rows (x within a halo); returns the thread's
// partial sum of x'y.  In single precision the CTAs take segments in turn: the
// grid sweeps the matrix as one front, so the values and the vector elements
// that a row max(off) further on reads again are still in L2, which they had
// left when each CTA swept a range of its own (108 000 rows at 256^3; 300 ->
// 240 us per reliable-update iteration).  In double precision, bound by the
// FP64 pipe, the even ranges [r0, r1) are 2-5% faster.
template <typename V, bool SYM>
__device__ __forceinline__ V dia_sweep(const DiaTab<V>& t, int64_t r0, int64_t r1, const V* x, V* y) {
  V dot = V(0);
  if constexpr (sizeof(V) == 8) {
    dia_rows<SYM, true, dia_c<V>(), dia_r<V>()>(t, (int)r0, (int)r1, x, [&](int i, V q) {
      y[i] = q;
      dot = dia_fma(x[i], q, dot);
    });
  } else {
    constexpr int R = dia_r<V>();
    const int lane = threadIdx.x & 31, per = blockDim.x * R;
    for (int64_t b = (int64_t)blockIdx.x * per + (threadIdx.x >> 5) * 32 * R; b < t.n; b += (int64_t)gridDim.x * per) {
      const int base = (int)b;
      V acc[R];
      dia_segment<SYM, false, true, dia_c<V>(), R>(t.entries(), t.K, t.lo, t.hi, t.val, t.n, t.n - 1, base, x, acc);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int i = base + lane + 32 * r;
        if (i < t.n) {
          y[i] = acc[r];
          dot = dia_fma(x[i], acc[r], dot);
        }
      }
    }
  }
  return dot;
}

// y = A x, R rows per thread, C diagonals in flight.
template <typename V, bool SYM, int R, int C>
__global__ void __launch_bounds__(kDiaBlock) k_dia_rows(const __grid_constant__ DiaDev<V> A, const V* __restrict__ x,
                                                       V* __restrict__ y) {
  const int base = (int)((blockIdx.x * (kDiaBlock / 32) + (threadIdx.x >> 5)) * 32 * R), n = (int)A.n;
  if (base >= n) return;
  V acc[R];
  dia_segment<SYM, true, false, C, R>(DiaParam<V>{A}, A.K, A.lo, A.hi, A.val, n, n - 1, base, x, acc);
  const int i0 = base + (threadIdx.x & 31);
#pragma unroll
  for (int r = 0; r < R; ++r)
    if (i0 + 32 * r < n) y[i0 + 32 * r] = acc[r];
}

}  // namespace gbcg
