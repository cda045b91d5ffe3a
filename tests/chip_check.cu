// chip_check.cu -- the scalar arithmetic of the solvers' steps (fp64.cuh) and
// the grid sums of the on-chip solvers (chip_solve.cuh), called by
// tests/test_scalars_host.py (host entries) and tests/test_gpu_scalars.py
// (device entries).
#include <cstdint>

#include "../paper_1010_4639_gb300/csrc/chip_solve.cuh"

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

constexpr int kSumThreads = 64;
// One grid sum per case: CTA c's partial sum is part[case * G + c], on one of
// its threads.  out and retaken (1: not the fixed-point sum) per case and CTA;
// absent: that CTA stays away, and ok tells what the others saw.
__global__ void k_sums(ChipSync* sync, const double* part, const double* prev, double* out, int32_t* retaken,
                       int32_t* ok, int cases, int absent, long long timeout_ns) {
  __shared__ double buf[kSumThreads + kMaxSums + 1];
  __shared__ int sok;
  __shared__ unsigned long long base[4];
  const int c = blockIdx.x, G = gridDim.x, t = threadIdx.x;
  GridSum g;
  g.sync = sync;
  g.buf = buf;
  g.out = buf + kSumThreads;
  g.ok = &sok;
  g.target = 0;
  g.sums = g.fast = 0;
  g.base = base;
  g.timeout_ns = timeout_ns;
  if (t < 4) base[t] = 0;
  __syncthreads();
  if (c == absent) return;
  for (int i = 0; i < cases; ++i) {
    const int before = g.sums;
    const bool fine = chip_sum_fast(g, t == i % kSumThreads ? part[(int64_t)i * G + c] : 0.0, prev[i],
                                    [](const double (&)[1]) {});
    if (t == 0) {
      ok[(int64_t)i * G + c] = fine;
      out[(int64_t)i * G + c] = g.out[0];
      retaken[(int64_t)i * G + c] = g.sums - before;
    }
    if (!fine) return;
    __syncthreads();
  }
}
}  // namespace

extern "C" {
// the sum of G partial sums by the words of chip_sum_fast; 1: it would be taken again
int host_fixed_sum(const double* part, int G, double prev, double* out) {
  const int ep = (int)((int64_t)double_bits(prev) >> 52);
  uint64_t hi = 12345, lo = 1ull << 63;  // what earlier sums left in the words
  const uint64_t hi0 = hi, lo0 = lo;
  for (int i = 0; i < G; ++i) {
    const FixedParts f = fixed_parts(part[i], ep);
    hi += ((uint64_t)f.hi << 8) + 1;
    lo += ((uint64_t)f.lo << 8) + 1;
  }
  if (((hi - hi0) & 255) != (uint64_t)G || ((lo - lo0) & 255) != (uint64_t)G) return -1;
  bool again;
  *out = fixed_value(FixedParts{(int64_t)(hi - hi0 - G) >> 8, (lo - lo0 - G) >> 8}, ep, again);
  return again;
}
// device arrays but sync_status (host); 0 or the CUDA error
int gpu_sums(const double* part, const double* prev, double* out, int32_t* retaken, int32_t* ok, int32_t cases,
             int32_t G, int32_t absent, int32_t timeout_ms, int32_t* sync_status) {
  ChipSync* sync = nullptr;
  cudaError_t e = cudaMalloc(&sync, sizeof(ChipSync));
  if (e == cudaSuccess) e = cudaMemset(sync, 0, sizeof(ChipSync));
  long long ns = timeout_ms * 1000000ll;
  void* args[] = {&sync, &part, &prev, &out, &retaken, &ok, &cases, &absent, &ns};
  if (e == cudaSuccess)
    e = cudaLaunchCooperativeKernel((const void*)k_sums, dim3(G), dim3(kSumThreads), args, 0, nullptr);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e == cudaSuccess) e = cudaMemcpy(sync_status, &sync->bar.status, 4, cudaMemcpyDeviceToHost);
  cudaFree(sync);
  return (int)e;
}
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
