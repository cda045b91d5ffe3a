// grad.cu -- the differentiable form of the solve.
//
// For a loss L(x) of the solution of A x = b, the adjoint solve
// A lambda = dL/dx (A symmetric: the same operator and the same solver)
// gives dL/db = lambda and dL/dA_ij = -lambda_i x_j.  The kernels here turn
// that into gradients of what the caller stores:
//   - k_grad_values: the sampled outer product on the stored pattern (one
//     value per stored entry; for symmetric storage an off-diagonal value
//     stands for A_ij and A_ji and gets both terms);
//   - k_element_grad: the chain rule through a finite-element assembly
//     A = sum_e coef_e Kh_e, given as stored positions and weights per element;
//   - k_assemble: that assembly, per stored position, summing its
//     contributions in a fixed order (no atomics, bitwise reproducible).
// All three are streaming kernels bound by HBM.
#include <cuda_runtime.h>

#include <algorithm>
#include <string>

#include "../../include/gbcg.h"

namespace gbcg {
void set_last_error(const std::string& m);
}

namespace {

int fail(int code, const std::string& msg) {
  gbcg::set_last_error(msg);
  return code;
}

constexpr int kLanesPerRow = 8;

// One group of 8 lanes per row (CSR / symmetric) or column (CSC) of the
// stored pattern; entries of the row are taken 8 at a time, so a group's
// stores are contiguous.
template <int FMT>
__global__ void __launch_bounds__(256) k_grad_values(int64_t n, const int32_t* __restrict__ ptr,
                                                     const int32_t* __restrict__ idx, int32_t base,
                                                     const double* __restrict__ lam, const double* __restrict__ x,
                                                     double* __restrict__ g) {
  const int sub = threadIdx.x % kLanesPerRow;
  const int64_t groups = (int64_t)gridDim.x * (blockDim.x / kLanesPerRow);
  for (int64_t r = (int64_t)blockIdx.x * (blockDim.x / kLanesPerRow) + threadIdx.x / kLanesPerRow; r < n;
       r += groups) {
    const double lr = lam[r], xr = x[r];
    const int64_t k1 = (int64_t)ptr[r + 1] - base;
    for (int64_t k = (int64_t)ptr[r] - base + sub; k < k1; k += kLanesPerRow) {
      const int64_t c = (int64_t)idx[k] - base;
      double v;
      if (FMT == GBCG_CSC)
        v = -(lam[c] * xr);  // column r, row c
      else if (FMT == GBCG_SYM_CSR_UPPER && c != r)
        v = -(lr * x[c] + lam[c] * xr);
      else
        v = -(lr * x[c]);
      g[k] = v;
    }
  }
}

// The two assembly kernels read a map of one position (or element number) and
// one weight per contribution, some 24 of them per unknown.  A thread that
// walks its own contributions from global memory touches a line of its own
// with every load (a warp's load then takes 32 cycles of L1), waits for each
// gather before the next, and on k_assemble idles while the one diagonal entry
// of the warp sums its 24 contributions (on GB300 an FP64 instruction occupies
// the pipe for 16 cycles whether 1 or 32 lanes take part).  So a block brings
// a run of contributions, weight and gathered value, into shared memory with
// contiguous loads, and each output is then summed from there by one thread,
// in the map's order.  Bounds: the map read once (12 bytes per
// contribution) and one FP64 FMA each.
constexpr int kGradThreads = 256;
constexpr int kStage = 2048;  // contributions staged at a time (16 bytes each)
constexpr int kPer = kStage / kGradThreads;

// A thread's contributions of a run of `len` starting at tw, tn: every
// kGradThreads-th.
struct Contributions {
  int32_t n[kPer];
  double w[kPer];
  __device__ __forceinline__ void load(const int32_t* __restrict__ tn, const double* __restrict__ tw, int len) {
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int j = (int)threadIdx.x + u * kGradThreads;
      n[u] = -1;
      w[u] = 0.0;
      if (j < len) {
        n[u] = __ldcs(tn + j);
        w[u] = __ldcs(tw + j);
      }
    }
  }
};
constexpr int kGradBlocks = 6;  // blocks per SM that the stage leaves room for

// gc[e] = sum over k of w[e, k] g[pos[e, k]].  64^3 nodes, full storage (1.5 M
// elements of 16 pairs, 288 MB of map): 140 us with a thread per element, 97
// staged, 70 with the next run's map loaded into registers before the sums of
// the present one start (which the assembly below has no registers for: 124 us
// without, 160 with).
// Elements lie an odd number of 16-byte pairs apart, so eight lanes' reads of
// a step fall into different banks.
__global__ void __launch_bounds__(kGradThreads, 4) k_element_grad(int64_t ne, int m, int per, uint32_t inv,
                                                               const int32_t* __restrict__ pos,
                                                               const double* __restrict__ w,
                                                               const double* __restrict__ g,
                                                               double* __restrict__ gc) {
  extern __shared__ double2 stage[];
  const int ms = m | 1;
  const int64_t step = (int64_t)gridDim.x * per;
  auto elements = [&](int64_t e0) { return (int)(ne - e0 < per ? ne - e0 : per); };
  Contributions c;
  int64_t e0 = (int64_t)blockIdx.x * per;
  if (e0 < ne) c.load(pos + e0 * m, w + e0 * m, elements(e0) * m);
  for (; e0 < ne; e0 += step) {
    const int cnt = elements(e0), len = cnt * m;
    double gv[kPer];
#pragma unroll
    for (int u = 0; u < kPer; ++u) gv[u] = c.n[u] >= 0 ? __ldg(g + c.n[u]) : 0.0;
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int j = (int)threadIdx.x + u * kGradThreads;
      const int e = (int)(((uint32_t)j * inv) >> 20);  // j / m
      // no position: -0.0 * 0.0 leaves the sum as it is
      if (j < len) stage[e * ms + (j - e * m)] = make_double2(c.n[u] >= 0 ? c.w[u] : -0.0, gv[u]);
    }
    __syncthreads();
    if (e0 + step < ne) c.load(pos + (e0 + step) * m, w + (e0 + step) * m, elements(e0 + step) * m);
    for (int e = threadIdx.x; e < cnt; e += kGradThreads) {
      double s = 0.0;
#pragma unroll 4
      for (int k = 0; k < m; ++k) {
        const double2 t = stage[e * ms + k];
        s = fma(t.x, t.y, s);
      }
      gc[e0 + e] = s;
    }
    __syncthreads();
  }
}

// val[p] = sum over k in [tptr[p], tptr[p + 1]) of tw[k] coef[telem[k]], 256
// positions per block.  The block's threads take its positions in order of
// their numbers of contributions, so that the 32 sums of a warp are about
// equally long.  64^3 nodes, full storage (3.5 M positions, 23 M
// contributions): 190 us with a thread per position, 124 so.
__global__ void __launch_bounds__(kGradThreads) k_assemble(int64_t nnz, const int64_t* __restrict__ tptr,
                                                           const int32_t* __restrict__ telem,
                                                           const double* __restrict__ tw,
                                                           const double* __restrict__ coef, double* __restrict__ val) {
  constexpr int kBins = 32;
  __shared__ double2 stage[kStage];
  __shared__ int64_t ptr[kGradThreads + 1];
  __shared__ int bin[kBins];
  __shared__ uint8_t order[kGradThreads];
  const int t = threadIdx.x;
  for (int64_t p0 = (int64_t)blockIdx.x * kGradThreads; p0 < nnz; p0 += (int64_t)gridDim.x * kGradThreads) {
    const int cnt = (int)(nnz - p0 < kGradThreads ? nnz - p0 : kGradThreads);
    for (int i = t; i <= cnt; i += kGradThreads) ptr[i] = tptr[p0 + i];
    if (t < kBins) bin[t] = 0;
    __syncthreads();
    // a counting sort by number of contributions (ties in any order: it only
    // decides which thread sums which position)
    const int64_t n0 = t < cnt ? ptr[t + 1] - ptr[t] : 0;
    // (a decreasing pointer is a position without contributions)
    const int b = n0 < 0 ? 0 : n0 < kBins ? (int)n0 : kBins - 1;
    const int rank = t < cnt ? atomicAdd(&bin[b], 1) : 0;
    __syncthreads();
    if (t < kBins) {
      const int own = bin[t];
      int sum = own;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int up = __shfl_up_sync(0xffffffffu, sum, o);
        if (t >= o) sum += up;
      }
      bin[t] = sum - own;
    }
    __syncthreads();
    if (t < cnt) order[bin[b] + rank] = (uint8_t)t;
    __syncthreads();
    const int mine = t < cnt ? order[t] : -1;
    const int64_t k0 = mine >= 0 ? ptr[mine] : 0, k1 = mine >= 0 ? ptr[mine + 1] : 0;
    double s = 0.0;
    for (int64_t c0 = ptr[0], end = ptr[cnt]; c0 < end; c0 += kStage) {
      const int len = (int)(end - c0 < kStage ? end - c0 : kStage);
#pragma unroll 4
      for (int j = t; j < len; j += kGradThreads)
        stage[j] = make_double2(__ldcs(tw + c0 + j), __ldg(coef + __ldcs(telem + c0 + j)));
      __syncthreads();
      const int a = (int)(k0 < c0 ? 0 : k0 - c0 < len ? k0 - c0 : len);
      const int z = (int)(k1 < c0 ? 0 : k1 - c0 < len ? k1 - c0 : len);
#pragma unroll 2
      for (int j = a; j < z; ++j) s = fma(stage[j].x, stage[j].y, s);
      __syncthreads();
    }
    if (mine >= 0) val[p0 + mine] = s;
    __syncthreads();  // ptr, bin and order are rewritten
  }
}

int grid_for(int64_t items, int per_block, int blocks_per_sm = 8) {
  int dev = 0, sms = 148;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t want = (items + per_block - 1) / per_block;
  const int64_t cap = (int64_t)sms * blocks_per_sm;
  return (int)(want < 1 ? 1 : (want < cap ? want : cap));
}

int launched(const char* what) {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(GBCG_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
  return GBCG_OK;
}

}  // namespace

extern "C" {

int gbcg_grad_values(int32_t format, int64_t n, int64_t nnz, const int32_t* ptr, const int32_t* idx,
                     int32_t index_base, const double* lambda, const double* x, double* grad, void* stream) {
  gbcg::set_last_error("");
  if (format != GBCG_CSR && format != GBCG_SYM_CSR_UPPER && format != GBCG_CSC)
    return fail(GBCG_ERR_INVALID, "unknown format");
  if (n < 0 || nnz < 0) return fail(GBCG_ERR_INVALID, "n and nnz must be non-negative");
  if (index_base != 0 && index_base != 1) return fail(GBCG_ERR_INVALID, "index_base must be 0 or 1");
  if (n == 0) return GBCG_OK;
  if (!ptr || !lambda || !x || (nnz > 0 && (!idx || !grad))) return fail(GBCG_ERR_INVALID, "null argument");
  cudaStream_t s = (cudaStream_t)stream;
  const int blocks = grid_for(n, 256 / kLanesPerRow);
  if (format == GBCG_CSR)
    k_grad_values<GBCG_CSR><<<blocks, 256, 0, s>>>(n, ptr, idx, index_base, lambda, x, grad);
  else if (format == GBCG_CSC)
    k_grad_values<GBCG_CSC><<<blocks, 256, 0, s>>>(n, ptr, idx, index_base, lambda, x, grad);
  else
    k_grad_values<GBCG_SYM_CSR_UPPER><<<blocks, 256, 0, s>>>(n, ptr, idx, index_base, lambda, x, grad);
  return launched("k_grad_values");
}

int gbcg_element_grad(int64_t ne, int32_t m, const int32_t* pos, const double* w, const double* grad,
                      double* grad_coef, void* stream) {
  gbcg::set_last_error("");
  if (ne < 0 || m < 0 || m > 64) return fail(GBCG_ERR_INVALID, "ne must be >= 0 and m in [0, 64]");
  if (ne == 0) return GBCG_OK;
  if (!grad_coef || (m > 0 && (!pos || !w || !grad))) return fail(GBCG_ERR_INVALID, "null argument");
  // elements per block: what the stage holds, at most one per thread; j / m =
  // (j inv) >> 20 for j < 2^20 / m
  const int per = m > 0 ? std::min(kGradThreads, kStage / (m | 1)) : kGradThreads;
  const uint32_t inv = m > 0 ? ((1u << 20) + m - 1) / m : 0;
  k_element_grad<<<grid_for(ne, per, 4), kGradThreads, sizeof(double2) * per * (m | 1), (cudaStream_t)stream>>>(
      ne, m, per, inv, pos, w, grad, grad_coef);
  return launched("k_element_grad");
}

int gbcg_assemble(int64_t nnz, const int64_t* tptr, const int32_t* telem, const double* tw, const double* coef,
                  double* val, void* stream) {
  gbcg::set_last_error("");
  if (nnz < 0) return fail(GBCG_ERR_INVALID, "nnz must be >= 0");
  if (nnz == 0) return GBCG_OK;
  if (!tptr || !val || !telem || !tw || !coef) return fail(GBCG_ERR_INVALID, "null argument");
  k_assemble<<<grid_for(nnz, kGradThreads, kGradBlocks), kGradThreads, 0, (cudaStream_t)stream>>>(nnz, tptr, telem, tw, coef, val);
  return launched("k_assemble");
}

}  // extern "C"
