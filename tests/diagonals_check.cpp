// diagonals_check.cpp -- host-side check of the diagonal layout (layout.cpp,
// build_diagonals), run by tests/test_diagonals_host.py without a GPU.  Reads
// a matrix (0-based arrays of the given format) from a binary file and prints
// NODIAGONALS when the layout's rule turns it down; otherwise checks that
//   - offsets are increasing, within the caps, and (symmetric) start at 0;
//   - every stored entry sits at its place with its value (zeros as +0.0) and
//     every other position holds -0.0;
// then runs the kernels' row sums (same order, same skips) in double
// precision and writes y after the input, for the caller to compare.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <string>
#include <vector>

#include "../paper_1010_4639_gb300/csrc/layout.h"

using namespace gbcg;

static int fail(const char* what, long long a = -1, long long b = -1) {
  printf("FAIL %s %lld %lld\n", what, a, b);
  return 1;
}
static bool padding(double v) { return v == 0.0 && std::signbit(v); }

int main(int argc, char** argv) {
  if (argc < 5) return fail("usage: diagonals_check matrix.bin format index_base y.bin");
  const int format = atoi(argv[2]), base = atoi(argv[3]);
  FILE* f = fopen(argv[1], "rb");
  if (!f) return fail("open");
  int64_t n = 0, nnz = 0;
  if (fread(&n, 8, 1, f) != 1 || fread(&nnz, 8, 1, f) != 1) return fail("header");
  std::vector<int32_t> ptr(n + 1), idx(nnz);
  std::vector<double> val(nnz), x(n), y(n);
  if (fread(ptr.data(), 4, n + 1, f) != (size_t)(n + 1) || fread(idx.data(), 4, nnz, f) != (size_t)nnz ||
      fread(val.data(), 8, nnz, f) != (size_t)nnz || fread(x.data(), 8, n, f) != (size_t)n)
    return fail("body");
  fclose(f);
  std::string err;
  if (validate_input(format, n, nnz, ptr.data(), idx.data(), val.data(), base, err)) return fail(err.c_str());
  DiaHost D;
  if (!build_diagonals(format, n, nnz, ptr.data(), idx.data(), val.data(), base, D)) {
    if (!D.val.empty() && D.off.empty()) return fail("not left empty");
    printf("NODIAGONALS\n");
    return 0;
  }
  const int K = (int)D.off.size();
  if (K < 1 || K > kMaxDiag || D.ld < n || D.ld % 64 || (int64_t)D.val.size() != K * D.ld) return fail("shape");
  for (int k = 1; k < K; ++k)
    if (D.off[k] <= D.off[k - 1]) return fail("offsets", k);
  if (format == 1 && D.off[0] != 0) return fail("diagonal first");
  if (3 * nnz < 2 * K * n) return fail("rule");
  std::vector<char> seen(D.val.size(), 0);
  for (int64_t l = 0; l < n; ++l)
    for (int64_t q = ptr[l] - base; q < ptr[l + 1] - base; ++q) {
      const int64_t r = format == 2 ? idx[q] - base : l, c = format == 2 ? l : idx[q] - base;
      int k = 0;
      while (k < K && D.off[k] != c - r) ++k;
      if (k == K) return fail("missing offset", r, c);
      const double v = D.val[k * D.ld + r];
      if (padding(v) || v != val[q]) return fail("value", r, c);
      seen[k * D.ld + r] = 1;
    }
  for (size_t i = 0; i < seen.size(); ++i)
    if (!seen[i] && !padding(D.val[i])) return fail("padding", (long long)i);
  for (int64_t i = 0; i < n; ++i) {
    auto term = [&](double& acc, int k, int64_t at, int64_t c) {
      if (c < 0 || c >= n) return;
      const double v = D.val[k * D.ld + at];
      if (!padding(v)) acc = std::fma(v, x[c], acc);
    };
    double acc = 0.0;
    if (format == 1)
      for (int k = K - 1; k >= 1; --k)
        if (i - D.off[k] >= 0) term(acc, k, i - D.off[k], i - D.off[k]);
    for (int k = 0; k < K; ++k) term(acc, k, i, i + D.off[k]);
    y[i] = acc;
  }
  f = fopen(argv[4], "wb");
  if (!f || fwrite(y.data(), 8, n, f) != (size_t)n) return fail("write");
  fclose(f);
  printf("OK diagonals %d\n", K);
  return 0;
}
