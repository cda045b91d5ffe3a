// fp64.cuh -- double-precision scalars on a GPU whose FP64 pipe is narrow.
// GB300 measured: an FP64 addition or FMA takes 64 cycles and occupies its SM
// sub-partition's pipe all that time, whether one lane takes part or 32 (16
// cycles of the SM per warp instruction); a division takes 657 cycles, a
// square root 688.  The helpers here keep them off the path between a
// reduction and the step that waits for it.
#pragma once
#include <cuda_runtime.h>

namespace gbcg {

// a / b, accurate to the rounding of V.  A reciprocal estimate with one Newton
// step gives a quotient within 2^-38, enough for a single-precision result;
// one correction by the quotient's residual makes it a double-precision one.
template <typename V>
__device__ __forceinline__ double quick_div(double a, double b) {
  const int ea = (__double2hiint(a) >> 20) & 0x7ff, eb = (__double2hiint(b) >> 20) & 0x7ff;
  if (ea < 128 || ea > 1918 || eb < 128 || eb > 1918) return a / b;  // near the ends of the range, 0, inf, NaN
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(b));
  r = fma(r, fma(-b, r, 1.0), r);
  const double q = a * r;
  return sizeof(V) == 4 ? q : fma(fma(-b, q, a), r, q);
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
