// fp64.cuh -- double-precision scalars on a GPU whose FP64 pipe is narrow.
// GB300 measured: an FP64 addition or FMA takes 64 cycles and occupies its SM
// sub-partition's pipe all that time, whether one lane takes part or 32 (16
// cycles of the SM per warp instruction); a division takes 549 cycles, a
// square root 688.  The helpers here keep them off the path between a
// reduction and the step that waits for it.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>
#include <cuda_runtime.h>

namespace gbcg {

__host__ __device__ __forceinline__ uint64_t double_bits(double v) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(v);
#else
  uint64_t u;
  memcpy(&u, &v, sizeof u);
  return u;
#endif
}
__host__ __device__ __forceinline__ double bits_double(uint64_t u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)u);
#else
  double v;
  memcpy(&v, &u, sizeof v);
  return v;
#endif
}

// a / b, rounded as IEEE 754 asks, on the integer units.  Long division of the
// significands in radix 2^18 with the quotient digits taken from a rounded
// reciprocal of the divisor's leading bits (very-high-radix division: Wong and
// Flynn, IEEE Trans. Computers 41(8), 1992).  A digit's estimate is within
// 1/2 + 2^-4 of the exact one (rounding, the reciprocal's 2^-23, four roundings
// of 2^-24 or less, each times the digit's 2^18), so the remainder stays below
// the divisor and the next digit within 2^18; its 64-bit difference is exact
// although both terms overflow.  After three digits the quotient has 54
// fraction bits and the remainder's sign tells which way it is rounded; a tie
// cannot occur (a quotient of 54 significant bits times the divisor has more
// bits than the dividend).  274 cycles in a chain of divisions against 549 for
// a / b; a Newton reciprocal on the FP64 pipe took 231 for a quotient within
// 2^-38 and 370 for a double-precision one.  Zeros, subnormal numbers, negative numbers,
// infinities, NaN and quotients near the ends of the range take a / b.
__host__ __device__ __forceinline__ double quick_div(double a, double b) {
  const uint64_t ua = double_bits(a), ub = double_bits(b);
  const unsigned ea = (unsigned)(ua >> 52), eb = (unsigned)(ub >> 52);  // with the sign
  int e = (int)ea - (int)eb + 1023;
  if (ea - 1u >= 2046u || eb - 1u >= 2046u || (unsigned)(e - 2) > 2042u) return a / b;
  uint64_t ma = (ua & 0xfffffffffffffull) | (1ull << 52);
  const uint64_t mb = (ub & 0xfffffffffffffull) | (1ull << 52);
  if (ma < mb) {
    ma <<= 1;
    --e;
  }
  const float top = (float)(int32_t)(mb >> 24);
#ifdef __CUDA_ARCH__
  float inv;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"(top));
#else
  const float inv = 1.f / top;
#endif
  int64_t q = 1, r = (int64_t)(ma - mb);  // the first digit is 1
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float t = (float)(int32_t)(r >> 24) * inv * 262144.f;
#ifdef __CUDA_ARCH__
    const int32_t d = __float2int_rn(t);
#else
    const int32_t d = (int32_t)lrintf(t);
#endif
    q = q * 262144 + d;
    r = (int64_t)(((uint64_t)r << 18) - (uint64_t)((int64_t)d) * mb);
  }
  const uint64_t m = (uint64_t)(q + 2 - (r < 0)) >> 2;  // in [2^52, 2^53]
  return bits_double(((uint64_t)e << 52) + (m - (1ull << 52)));
}

// A comparison also runs on the FP64 pipe; the bits do not.
__device__ __forceinline__ bool quick_finite(double s) {
  return ((unsigned)__double2hiint(s) & 0x7ff00000u) != 0x7ff00000u;
}
__device__ __forceinline__ bool quick_positive(double s) { return __double_as_longlong(s) > 0; }  // of a finite s

// Tests sqrt(s) against a bound c without the square root: s is compared, as
// an integer, with c^2 a little enlarged and reduced; only in between does the
// exact test run.
struct SqrtTest {
  long long lo, hi;
  __device__ __forceinline__ void set(double c) {
    const double c2 = c * c;
    lo = 0;  // undecided everywhere
    hi = 0x7ff0000000000000ll;
    if (c2 > 1e-290 && c2 < 1e290) {
      lo = __double_as_longlong(c2 * (1.0 - 1e-12));
      hi = __double_as_longlong(c2 * (1.0 + 1e-12));
    }
  }
  // s >= 0 and finite; exact() decides in between
  template <class X>
  __device__ __forceinline__ bool below(double s, X&& exact) const {
    const long long b = __double_as_longlong(s);
    return b < lo ? true : b > hi ? false : exact();
  }
};

// (double)f for the FP64 pipe's sake: a normal number's bits are moved.
__device__ __forceinline__ double quick_double(float f) {
  const unsigned b = __float_as_uint(f), e = (b >> 23) & 0xffu;
  if (e - 1u >= 254u) return f == 0.f ? __hiloint2double((int)(b & 0x80000000u), 0) : (double)f;
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
}
__device__ __forceinline__ double quick_double(double f) { return f; }

}  // namespace gbcg
