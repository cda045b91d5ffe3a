// chip_check.cu -- the scalar arithmetic of the solvers' steps (fp64.cuh),
// called by tests/test_scalars_host.py (host entries) and
// tests/test_gpu_scalars.py (device entries).
#include <cstdint>

#include "../paper_1010_4639_gb300/csrc/fp64.cuh"

using namespace gbcg;

namespace {
__global__ void k_div(const double* a, const double* b, double* q, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    q[i] = quick_div(a[i], b[i]);
}
__global__ void k_widen(const float* f, double* d, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    d[i] = quick_double(f[i]);
}
// bit 0: quick_finite, 1: quick_positive, 2: below(s) by SqrtTest, 3: sqrt(s) <= c
__global__ void k_tests(const double* s, const double* c, int32_t* out, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    SqrtTest t;
    t.set(c[i]);
    const bool exact = sqrt(s[i]) <= c[i], below = t.below(s[i], [&] { return exact; });
    out[i] = (quick_finite(s[i]) ? 1 : 0) | (quick_positive(s[i]) ? 2 : 0) | (below ? 4 : 0) | (exact ? 8 : 0);
  }
}
}  // namespace

extern "C" {
void host_div(const double* a, const double* b, double* q, int64_t n) {
  for (int64_t i = 0; i < n; ++i) q[i] = quick_div(a[i], b[i]);
}
// device arrays; 0 or the CUDA error
int gpu_div(const double* a, const double* b, double* q, int64_t n) {
  k_div<<<608, 256>>>(a, b, q, n);
  return (int)cudaDeviceSynchronize();
}
int gpu_widen(const float* f, double* d, int64_t n) {
  k_widen<<<608, 256>>>(f, d, n);
  return (int)cudaDeviceSynchronize();
}
int gpu_tests(const double* s, const double* c, int32_t* out, int64_t n) {
  k_tests<<<608, 256>>>(s, c, out, n);
  return (int)cudaDeviceSynchronize();
}
}
