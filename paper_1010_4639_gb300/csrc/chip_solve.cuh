// chip_solve.cuh -- the persistent conjugate-gradient solvers whose vectors
// stay on the chip, on the diagonal layout and, for short ranges of rows per
// CTA, on the row-gather layout.
//
// One CTA per SM owns a contiguous range of rows and keeps those rows of x,
// r, p and q = A p in shared memory for the whole solve; thread t owns rows
// t, t + T, ... of the range, so the vector updates need no synchronisation
// at all.  Only what other CTAs read goes to global memory.  An iteration is
//   A: q = A p, p'q                                     -> grid sum
//   B: x += alpha p, r -= alpha q (on chip), r'r        -> grid sum
//   C: p = r + beta p (on chip, and out to global memory) -> grid barrier
// (Forming p = r + beta p in A at every column a row reads, from r and the
// previous p in global memory, saves C's barrier but loads twice as much: no
// faster at 25 000 rows, 20% slower per iteration at 238 000.)
//
// The arithmetic is that of k_cg and k_cg_ru (kernels.cuh), step by step.
#pragma once
#include "fp64.cuh"
#include "kernels.cuh"

namespace gbcg {

// Threads per CTA, at most (fewer when a CTA owns fewer rows), by rows per
// thread and product step.
constexpr int kChipThreads = 1024;
constexpr int chip_threads(int R) { return R == 1 ? 512 : kChipThreads; }
constexpr int kMaxSums = 3;         // values per grid sum
constexpr int kSumLanes = 8;        // partial sums per lane of warp 0: up to 256 CTAs

// Device words of one handle's solver: the barrier, then the partial sums
// (two sets, used in turn: a CTA can be one sum ahead of another).
// acc: the fixed-point sums of chip_sum_fast, high and low words on lines of
// their own.
struct ChipSync {
  GridBar bar;
  double part[2][kMaxSums][32 * kSumLanes];
  alignas(128) unsigned long long acc[2][2][16];
};
constexpr int kChipCtas = 255;  // chip_sum_fast counts arrivals in 8 bits

// State of the grid sums of one launch.
struct GridSum {
  ChipSync* sync;
  double* buf;                // shared memory: blockDim.x partial sums
  double* out;                // shared memory: the sums
  int* ok;                    // shared memory
  unsigned long long target;  // arrivals at the barrier's counter
  unsigned long long* base;   // shared memory: words of the last two fast sums, [2][2]
  int sums, fast;             // sums done
  long long timeout_ns;
};

// Sums NV values over every thread of the grid, in a fixed order, and is a
// grid barrier.  f(sums) then runs on thread 0 before the CTA goes on (the
// step's scalars).  False, uniformly within the CTA, when a wait ran out or
// another CTA failed.
//
// FP64 additions are slow (fp64.cuh), useful lanes or not, so the CTA's
// partial sums go through shared memory and are added by one warp (four when
// there are many) instead of a shuffle tree in every warp.  Measured with 152
// CTAs: an arrival at one counter that a warp per CTA polls costs 2 600
// cycles; flags polled all-to-all, with the sums in them, 4 400 to 8 000.
template <int NV>
__device__ __forceinline__ void chip_cta_sum(GridSum& g, const double (&v)[NV], double (&s)[NV]) {
  const int t = threadIdx.x, T = blockDim.x;
#pragma unroll
  for (int j = 0; j < NV; ++j) {
    if (j > 0) __syncthreads();
    g.buf[t] = v[j];
    __syncthreads();  // every thread's partial sum (and, for the first, its global writes)
    if (T > 256 && t < 128) {
      double x = g.buf[t];
      for (int i = t + 128; i < T; i += 128) x += g.buf[i];
      g.buf[t] = x;
      asm volatile("bar.sync 1, 128;" ::: "memory");
    }
    if (t < 32) {
      const int m = T > 256 ? 128 : T;
      s[j] = g.buf[t];
      for (int i = t + 32; i < m; i += 32) s[j] += g.buf[i];
#pragma unroll
      for (int o = 16; o; o >>= 1) s[j] += __shfl_xor_sync(0xffffffffu, s[j], o);
    }
  }
}

template <int NV, class F>
__device__ __forceinline__ bool chip_sum(GridSum& g, const double (&v)[NV], F&& f) {
  const int t = threadIdx.x, G = gridDim.x, lane = t & 31;
  g.target += G;
  double(*part)[32 * kSumLanes] = g.sync->part[++g.sums & 1];
  double s[NV];
  chip_cta_sum(g, v, s);
  if (t < 32) {
    if (lane == 0) {
#pragma unroll
      for (int j = 0; j < NV; ++j) __stcg(&part[j][blockIdx.x], s[j]);
      red_release_add(&g.sync->bar.count, 1ull);
    }
    __syncwarp();
    bool ok = true;
    long long t0 = 0;
    for (unsigned spins = 1; ld_acquire(&g.sync->bar.count) < g.target; ++spins)  // the warp polls one word
      if ((spins & 63u) == 0) {
        if (t0 == 0) t0 = gtime();
        if (ld_relaxed(&g.sync->bar.status) != 0) ok = false;
        else if (gtime() - t0 > g.timeout_ns) {
          if (atomicCAS(&g.sync->bar.status, 0, (int)kTimeout) == 0) g.sync->bar.where = g.sums;
          ok = false;
        }
        if (!ok) break;
      }
    ok = __all_sync(0xffffffffu, ok);
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      double w[kSumLanes];
#pragma unroll
      for (int u = 0; u < kSumLanes; ++u) w[u] = lane + 32 * u < G ? __ldcg(&part[j][lane + 32 * u]) : 0.0;
      double x = w[0];
#pragma unroll
      for (int u = 1; u < kSumLanes; ++u)
        if (32 * u < G) x += w[u];
#pragma unroll
      for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      s[j] = x;
    }
    if (lane == 0) {
#pragma unroll
      for (int j = 0; j < NV; ++j) g.out[j] = s[j];
      *g.ok = ok;
      if (ok) f(s);
    }
  }
  __syncthreads();
  return *g.ok != 0;
}
template <int NV>
__device__ __forceinline__ bool chip_sum(GridSum& g, const double (&v)[NV]) {
  return chip_sum<NV>(g, v, [](const double (&)[NV]) {});
}
__device__ __forceinline__ bool chip_barrier(GridSum& g) {
  return grid_barrier(&g.sync->bar, g.target, g.timeout_ns, g.ok, g.sums);
}

// A CTA's partial sum as a fixed-point number whose unit is 2^-72 of the
// leading bit of `prev` (ep: prev's sign and exponent): 40 low bits, and a
// signed high part of 47.  kFixMark as the low part when it does not fit
// (2^15 of prev and above, infinities, NaN).
constexpr int kFixUnit = 72;  // unit below prev, in bits
constexpr int kFixFall = 10;  // a sum may be this many bits below prev
constexpr unsigned long long kFixMark = 1ull << 48;
struct FixedParts {
  long long hi;
  unsigned long long lo;
};
__host__ __device__ __forceinline__ FixedParts fixed_parts(double s, int ep) {
  const unsigned long long bits = double_bits(s);
  const int es = (int)(bits >> 52) & 0x7ff, sh = es - ep + kFixUnit - 52;
  const unsigned long long m = (bits & 0xfffffffffffffull) | (1ull << 52), low40 = (1ull << 40) - 1;
  FixedParts f = {0, 0};
  if (sh > 34) {
    f.lo = kFixMark;
  } else if (es > 0 && sh > -53) {
    const unsigned long long w = sh < 0 ? m >> -sh : m;
    const int up = sh < 0 ? 0 : sh;
    f.lo = (w << up) & low40;
    f.hi = (long long)(w >> (40 - up));
    if ((long long)bits < 0) {
      f.hi = f.lo ? -f.hi - 1 : -f.hi;
      f.lo = (0 - f.lo) & low40;
    }
  }
  return f;
}
// The sum of such parts as a double; `again`: it was marked, or is less than
// 2^-10 of prev (or negative), where the parts' truncations would count.
__host__ __device__ __forceinline__ double fixed_value(FixedParts sum, int ep, bool& again) {
  const double unit = bits_double((uint64_t)(ep - kFixUnit) << 52);  // powers of two scale exactly
  const double v = fma((double)sum.hi, unit * 0x1p40, (double)(long long)sum.lo * unit);
  again = sum.lo >= kFixMark || (int)((long long)double_bits(v) >> 52) < ep - kFixFall;
  return v;
}

// chip_sum of one value per thread whose sum is expected within 2^-10 .. 2^14
// of `prev` (the same sum an iteration earlier), without a memory fence: it
// orders nothing but the sum itself.  Each CTA adds its partial sum to two
// 64-bit integers with relaxed atomics, as a fixed-point number (fixed_parts),
// and each word counts its arrivals in its low 8 bits; a CTA polls the two
// words until both counts are full and has the sum.  Integer addition makes
// the sum independent of the order of arrival, and exact but for the parts'
// truncations, less than one unit each: below 2^(8 - 72 + 10) = 2^-54 of the
// smallest sum taken, a quarter of its last bit, before its rounding to double
// precision.  (With a unit of 2^-67 and sums down to 2^-13 it was 2^-46.)
// This replaces a store of the partial sum, the fence that publishes it, a
// poll, a load of all partial sums and their additions: 5 100 -> 2 900 cycles
// per sum with 152 CTAs.  A marked or unexpectedly small sum is taken again by
// chip_sum, by every CTA alike.
template <class F>
__device__ __forceinline__ bool chip_sum_fast(GridSum& g, double v, double prev, F&& step) {
  const int t = threadIdx.x, lane = t & 31;
  const int ep = __double2hiint(prev) >> 20;  // sign and exponent
  const double v1[1] = {v};
  if (ep < 256 || ep > 1790) return chip_sum<1>(g, v1, step);
  const unsigned G = gridDim.x;
  const int set = ++g.fast & 1;
  double s1[1];
  chip_cta_sum(g, v1, s1);
  if (t < 32) {
    const FixedParts f = fixed_parts(s1[0], ep);
    unsigned long long* word = g.sync->acc[set][lane & 1];
    unsigned long long* base = g.base + 2 * set + (lane & 1);
    unsigned long long w = 0;
    bool ok = true;
    if (lane < 2) {
      const unsigned long long add = ((lane ? f.lo : (unsigned long long)f.hi) << 8) + 1ull;
      asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(word), "l"(add) : "memory");
      const unsigned long long b0 = *base;
      long long t0 = 0;
      for (unsigned spins = 1;; ++spins) {
        asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(word) : "memory");
        if ((unsigned)((w - b0) & 255u) == G) break;
        if ((spins & 63u) == 0) {
          if (t0 == 0) t0 = gtime();
          if (ld_relaxed(&g.sync->bar.status) != 0) ok = false;
          else if (gtime() - t0 > g.timeout_ns) {
            if (atomicCAS(&g.sync->bar.status, 0, (int)kTimeout) == 0) g.sync->bar.where = 1000000 + g.fast;
            ok = false;
          }
          if (!ok) break;
        }
      }
      *base = w;
      w -= b0 + G;
    }
    __syncwarp();
    ok = __all_sync(0xffffffffu, ok);
    const unsigned long long wlo = __shfl_sync(0xffffffffu, w, 1) >> 8;
    if (lane == 0) {
      bool again;
      const double sum[1] = {fixed_value(FixedParts{(long long)w >> 8, wlo}, ep, again)};
      g.out[0] = sum[0];
      *g.ok = !ok ? 0 : again ? 2 : 1;
      if (ok && !again) step(sum);
    }
  }
  __syncthreads();
  if (*g.ok != 2) return *g.ok != 0;
  return chip_sum<1>(g, v1, step);
}

// What a solve does around its iterations: the double-precision solve from
// x0 with true-residual confirmation and restarts; the single-precision inner
// solve of the refinement (from 0, to a tolerance of its own); or
// single-precision iterations with double-precision reliable updates.
enum { kSolveFull = 0, kSolveInner = 1, kSolveRu = 2 };

template <typename V>
struct ChipArgs {
  DiaDev<V> D;         // kDia, kDiaSym
  DiaDev<double> D64;  // kSolveRu
  OpDev<V> A;          // kGather
  OpDev<double> A64;   // kSolveRu
  const int32_t* cta_slice;
  const int32_t* cta_long;
  V* x;                // kSolveFull: the caller's x; kSolveInner: the correction (out)
  const V* b;
  V* p;                // p in global memory
  double* x64;         // kSolveRu: the caller's x and b
  const double* b64;
  double* xh;          // kSolveRu: x within a halo, for the update's product
  ChipSync* sync;
  CgState* st;
  int32_t n;
  double tol, delta;
  int32_t maxit, max_restarts;
  int32_t rows;        // greatest number of rows of a CTA
  long long timeout_ns;
};

// Shared memory of a CTA: four vectors of its rows, the sums' buffers, the
// offsets of its slices (row gather).
template <typename V>
size_t chip_smem(int64_t rows, int threads) {
  return 4 * (size_t)rows * sizeof(V) + ((size_t)threads + kMaxSums + 1 + rows / 32 + 1) * sizeof(double);
}

// f(row, (A x)_row) over the slices of rows [r0, r1) (their offsets in shared
// memory) and the long rows [l0, l1) of the row-gather layout, straight from
// global memory: eight entries' columns and values, then their gathers, are
// in flight together.  The bulk-copy pipeline of spmv_rows keeps more bytes in
// flight over long ranges; with one or two slices per warp its stage wait only
// adds to the chain.
template <typename V, class F>
__device__ __forceinline__ void chip_gather(const OpDev<V>& A, const int64_t* off, int r0, int r1, int l0, int l1,
                                            const V* x, F&& f) {
  constexpr int C = 8;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int s = warp; r0 + 32 * s < r1; s += nw) {
    const int64_t beg = off[s];
    const int L = (int)((off[s + 1] - beg) >> 5), row = r0 + 32 * s + lane;
    const V* __restrict__ val = A.val + beg + lane;
    V acc = V(0);
    auto terms = [&](auto* __restrict__ col, const V* xb) {
      for (int k0 = 0; k0 < L; k0 += C) {
        V v[C], xv[C];
        int c[C];
#pragma unroll
        for (int j = 0; j < C; ++j) {
          const int k = min(k0 + j, L - 1);
          c[j] = __ldg(col + 32 * k);
          v[j] = __ldg(val + 32 * k);
        }
#pragma unroll
        for (int j = 0; j < C; ++j) xv[j] = xb[c[j]];
#pragma unroll
        for (int j = 0; j < C; ++j)
          if (k0 + j < L) acc = dia_fma(v[j], xv[j], acc);
      }
    };
    // 16-bit offsets count from the row (lanes past the last row read x[0])
    if (A.col16) terms(A.col16 + beg + lane, x + (row < r1 ? row : 0));
    else terms(A.col + beg + lane, x);
    if (row < r1 && !((A.long_mask[(r0 >> 5) + s] >> lane) & 1u)) f(row, acc);
  }
  for (int li = l0 + warp; li < l1; li += nw) {
    const V v = long_row<V, false>(A, li, lane, x);
    if (lane == 0) f((int)A.long_row[li], v);
  }
}

// The matrix as a CTA sees it.
template <typename V, int FMT>
struct ChipMat {
  const DiaTab<V>& tab;
  const OpDev<V>& A;
  const int64_t* off;
  int r0, r1, l0, l1;
  template <bool HALO, int C, int R, class F>
  __device__ __forceinline__ void rows(const V* x, F&& f) const {
    if constexpr (is_dia(FMT)) dia_rows<FMT == kDiaSym, HALO, C, R>(tab, r0, r1, x, f);
    else chip_gather(A, off, r0, r1, l0, l1, x, f);
  }
};

// kSolveRu: float(b - A x) of the CTA's rows in double precision, into sr; the
// thread's sums of the residual's square (before and after rounding) and b's.
// A function of its own: a dozen calls per solve, and its registers would
// crowd the iterations'.
template <typename V, int FMT>
__device__ __noinline__ void chip_residual64(const ChipMat<double, FMT>& M, const double* b, const double* x, V* sr,
                                             double* sums) {
  double tt = 0.0, bb = 0.0;
  V rr = V(0);
  M.template rows<true, 8, 1>(x, [&](int i, double q) {
    const double bi = b[i], ti = bi - q;
    const V tf = (V)ti;
    sr[i] = tf;
    tt = fma(ti, ti, tt);
    rr = dia_fma(tf, tf, rr);
    bb = fma(bi, bi, bb);
  });
  sums[0] = tt;
  sums[1] = (double)rr;
  sums[2] = bb;
}

template <typename V, int FMT, int KIND, int R>
__global__ void __launch_bounds__(chip_threads(R), 1) k_cg_chip(const __grid_constant__ ChipArgs<V> a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ DiaTab<V> tab;
  __shared__ DiaTab<double> tab64;
  __shared__ struct {
    double alpha, beta;
    int code;
  } sc;  // the step's scalars, formed by thread 0 as a grid sum ends
  __shared__ int sok;
  __shared__ unsigned long long sbase[4];
  const int c = blockIdx.x, t = threadIdx.x, T = blockDim.x;
  const int r0 = a.cta_slice[c] * 32, r1 = min(a.cta_slice[c + 1] * 32, a.n);
  constexpr int C = R == 1 ? 8 : 16 / (R * (int)sizeof(V));  // diagonals whose loads are in flight together
  GridSum g;
  g.sync = a.sync;
  g.buf = reinterpret_cast<double*>(smem_raw);
  g.out = g.buf + T;
  g.ok = &sok;
  g.target = 0;
  g.sums = g.fast = 0;
  g.base = sbase;
  if (t < 4) sbase[t] = 0;
  g.timeout_ns = a.timeout_ns;
  int64_t* off = reinterpret_cast<int64_t*>(g.out + kMaxSums + 1);
  V* sx = reinterpret_cast<V*>(off + a.rows / 32 + 1) - r0;  // indexed by row
  V* sr = sx + a.rows;
  V* sq = sr + a.rows;
  V* sp = sq + a.rows;
  const int l0 = FMT == kGather ? a.cta_long[c] : 0, l1 = FMT == kGather ? a.cta_long[c + 1] : 0;
  if constexpr (is_dia(FMT)) {
    dia_tab_init(tab, a.D);
    if constexpr (KIND == kSolveRu) dia_tab_init(tab64, a.D64);
  } else {
    for (int s = t; s <= (r1 - r0 + 31) / 32; s += T) off[s] = a.A.sl_ptr[r0 / 32 + s];
  }
  const ChipMat<V, FMT> M{tab, a.A, off, r0, r1, l0, l1};
  __syncthreads();
  int status = kOk, k = 0, restarts = 0;
  double rr = 0.0, nb = 0.0, rel = 0.0, rmax = 0.0, beta = 0.0, pq = 0.0;
  bool conv = false;
  SqrtTest at_tol, at_delta;

  // kSolveFull: r = b - A x from the x in global memory; returns r'r
  auto residual = [&](double& tt, double& bb) {
    V ptt = V(0), pbb = V(0);
    M.template rows<false, C, R>((const V*)a.x, [&](int i, V q) {
      const V bi = a.b[i];
      const V ri = bi - q;
      sr[i] = ri;
      ptt = dia_fma(ri, ri, ptt);
      pbb = dia_fma(bi, bi, pbb);
    });
    tt = (double)ptt;
    bb = (double)pbb;
  };
  // kSolveRu: x += d, d = 0; r = float(b - A64 x); rr = r'r, rel = ||b - A x|| / ||b||
  bool first_update = true;
  auto update = [&]() -> bool {
    for (int i = r0 + t; i < r1; i += T) {
      const double xi = a.x64[i] + (double)sx[i];
      a.x64[i] = xi;
      a.xh[i] = xi;
      sx[i] = V(0);
    }
    if (!chip_barrier(g)) return false;  // x of every CTA
    double v[3];
    const ChipMat<double, FMT> M64{tab64, a.A64, off, r0, r1, l0, l1};
    chip_residual64<V, FMT>(M64, a.b64, a.xh, sr, v);
    if (!chip_sum<3>(g, v)) return false;
    const double tt = g.out[0];
    rr = g.out[1];
    if (first_update) nb = sqrt(g.out[2]);
    first_update = false;
    rel = nb > 0.0 ? sqrt(tt) / nb : 0.0;
    rmax = sqrt(rr);
    at_delta.set(a.delta * rmax);
    return true;
  };
  // p = r + beta p of the CTA's rows, on the chip and out.  Another CTA may have
  // read the former p as the two sums since then order nothing in memory; but
  // what it read went into its part of p'q, which it could only publish once
  // the values were there, and this CTA has waited for every part.  (Reads
  // whose value is not used may see either p.)
  auto direction = [&]() -> bool {
    const V be = (V)beta;
    for (int i = r0 + t; i < r1; i += T) {
      const V pi = dia_fma(be, sp[i], sr[i]);
      sp[i] = pi;
      a.p[i] = pi;
    }
    return chip_barrier(g);
  };
  auto store_x = [&]() {
    if constexpr (KIND == kSolveRu) {
      for (int i = r0 + t; i < r1; i += T) a.x64[i] += (double)sx[i];
    } else {
      for (int i = r0 + t; i < r1; i += T) a.x[i] = sx[i];
    }
  };

  // p = r: beta = 0 with a zero p before it
  for (int i = r0 + t; i < r1; i += T) {
    sp[i] = V(0);
    sx[i] = V(0);
  }
  if constexpr (KIND == kSolveRu) {
    if (!update()) return;
    if (nb == 0.0) {  // b = 0: x = 0
      for (int i = r0 + t; i < r1; i += T) a.x64[i] = 0.0;
      rel = 0.0;
      goto finish;
    }
    if (!isfinite(rel)) {
      status = kNonfinite;
      goto finish;
    }
    if (rel <= a.tol) goto finish;
    status = kMaxit;
  } else {
    double v[2];
    if constexpr (KIND == kSolveFull) {
      residual(v[0], v[1]);
      for (int i = r0 + t; i < r1; i += T) sx[i] = a.x[i];
    } else {
      V prr = V(0);
      for (int i = r0 + t; i < r1; i += T) {
        const V bi = a.b[i];
        sr[i] = bi;
        prr = dia_fma(bi, bi, prr);
      }
      v[0] = v[1] = (double)prr;
    }
    if (!chip_sum<2>(g, v)) return;
    rr = g.out[0];
    nb = sqrt(g.out[1]);
    if (nb == 0.0) {  // b = 0: x = 0
      for (int i = r0 + t; i < r1; i += T) a.x[i] = V(0);
      rr = 0.0;
      goto finish;
    }
    conv = sqrt(rr) / nb <= a.tol;
  }
  at_tol.set(a.tol * nb);
  for (;;) {
    while (k < a.maxit && !conv) {
      // C of the step before (the first p is r)
      if (!direction()) return;
      // A: q = A p, p'q
      double v[1];
      {
        V ppq = V(0);
        M.template rows<true, C, R>((const V*)a.p, [&](int i, V q) {
          sq[i] = q;
          ppq = dia_fma(sp[i], q, ppq);
        });
        v[0] = quick_double(ppq);
      }
      if (!chip_sum_fast(g, v[0], pq, [&](const double (&s)[1]) {
            sc.code = !quick_finite(s[0]) ? kNonfinite : !quick_positive(s[0]) ? kNotSpd : kOk;
            sc.alpha = quick_div(rr, s[0]);
          }))
        return;
      pq = g.out[0];
      if (sc.code != kOk) {
        status = sc.code;
        break;
      }
      // B: x += alpha p, r -= alpha q, r'r
      {
        const V al = (V)sc.alpha;
        V prr = V(0);
        for (int i = r0 + t; i < r1; i += T) {
          sx[i] = dia_fma(al, sp[i], sx[i]);
          const V ri = dia_fma(-al, sq[i], sr[i]);
          sr[i] = ri;
          prr = dia_fma(ri, ri, prr);
        }
        v[0] = quick_double(prr);
      }
      // kSolveRu: an update comes first when the recurrence residual has fallen
      // by delta, has reached tol, or the iteration bound is met
      if (!chip_sum_fast(g, v[0], rr, [&](const double (&s)[1]) {
            const double z = s[0];
            if (!quick_finite(z)) {
              sc.code = 2;
            } else if constexpr (KIND == kSolveRu) {
              const bool fell = at_delta.below(z, [&] { return sqrt(z) < a.delta * rmax; });
              sc.code = fell || k + 1 >= a.maxit || at_tol.below(z, [&] { return sqrt(z) <= a.tol * nb; }) ? 1 : 0;
            } else {
              sc.code = at_tol.below(z, [&] { return sqrt(z) / nb <= a.tol; }) ? 1 : 0;
            }
            sc.beta = quick_div(z, rr);
          }))
        return;
      ++k;
      const double rr_old = rr;
      rr = g.out[0];
      beta = sc.beta;
      const int code = sc.code;
      if (code == 2) {
        status = kNonfinite;
        break;
      }
      if (code == 1) {
        if constexpr (KIND == kSolveRu) {
          if (!update()) return;
          ++restarts;
          if (!isfinite(rel)) {
            status = kNonfinite;
            goto finish;
          }
          if (rel <= a.tol) {
            status = kOk;
            goto finish;
          }
          if (k >= a.maxit) {
            status = kMaxit;
            goto finish;
          }
          beta = rr / rr_old;  // the replaced residual's r'r (set by update())
        } else {
          conv = true;
        }
      }
    }
    if constexpr (KIND == kSolveFull) {
      if (status != kOk) break;
      // confirm on the true residual; restart the recurrence from it otherwise
      store_x();
      if (!chip_barrier(g)) return;
      double v[2];
      residual(v[0], v[1]);
      if (!chip_sum<2>(g, v)) return;
      const double tt = g.out[0];
      rel = sqrt(tt) / nb;
      if (!isfinite(tt)) {
        status = kNonfinite;
        break;
      }
      if (rel <= a.tol) break;
      if (k >= a.maxit || restarts >= a.max_restarts) {
        status = kMaxit;
        break;
      }
      ++restarts;
      rr = tt;
      beta = 0.0;
      conv = sqrt(rr) / nb <= a.tol;
    } else {
      if (KIND == kSolveInner && status == kOk && !conv) status = kMaxit;
      break;
    }
  }
  store_x();
finish:
  if (c == 0 && t == 0) {
    a.st->rr = rr;
    a.st->nb = nb;
    a.st->rel_true = rel;
    a.st->k = k;
    a.st->restarts = restarts;
    a.st->status = status;
  }
}

}  // namespace gbcg
