// scattered_check.cpp -- host-side check of the row-gather layout that
// symmetric storage with scattered neighbours takes (layout.cpp,
// build_sym_full, sym_slices_fit), run by tests/test_scattered_host.py
// without a GPU.  Reads an upper triangle and a vector, prints the windows per
// tile, and checks that
//   - sym_slices_fit says what build_sym_tiles does with the same caps;
//   - entry counts are those of the general symmetric layout;
// then sums the rows as the kernels read them (padding has value 0 and the
// row's own column) and writes y.
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

int main(int argc, char** argv) {
  if (argc < 6) return fail("usage: scattered_check matrix.bin index_base slot_cap ent_cap y.bin");
  const int base = atoi(argv[2]), slot_cap = atoi(argv[3]), ent_cap = atoi(argv[4]);
  FILE* f = fopen(argv[1], "rb");
  int64_t n = 0, nnz = 0;
  if (!f || fread(&n, 8, 1, f) != 1 || fread(&nnz, 8, 1, f) != 1) return fail("header");
  std::vector<int32_t> ptr(n + 1), idx(nnz);
  std::vector<double> val(nnz), x(n), y(n, 0.0);
  if (fread(ptr.data(), 4, n + 1, f) != (size_t)(n + 1) || fread(idx.data(), 4, nnz, f) != (size_t)nnz ||
      fread(val.data(), 8, nnz, f) != (size_t)nnz || fread(x.data(), 8, n, f) != (size_t)n)
    return fail("body");
  fclose(f);
  std::string err;
  LayoutHost G, L;
  SymTilesHost T;
  if (build_layout(1, n, nnz, ptr.data(), idx.data(), val.data(), base, G, err)) return fail(err.c_str());
  const double windows = sym_windows(n, ptr.data(), idx.data(), base);
  const bool fits = sym_slices_fit(n, ptr.data(), idx.data(), base, slot_cap, ent_cap);
  if (fits != build_sym_tiles(G, 1, slot_cap, ent_cap, 15, T)) return fail("fits", fits);
  if (!build_sym_full(n, nnz, ptr.data(), idx.data(), val.data(), base, L)) return fail("full");
  if (L.n != n || L.nnz_input != G.nnz_input || L.nnz_full != G.nnz_full) return fail("counts", L.nnz_full, G.nnz_full);
  const SellHost& A = L.A;
  for (int64_t r = 0; r < n; ++r) {
    const int64_t s = r / 32, l = r % 32;
    if (A.long_mask[s] >> l & 1) continue;
    for (int64_t at = A.sl_ptr[s] + l; at < A.sl_ptr[s + 1]; at += 32) {
      if (A.col[at] < 0 || A.col[at] >= n) return fail("column", r, A.col[at]);
      if (!A.col16.empty() && r + A.col16[at] != A.col[at]) return fail("16-bit column", r, A.col[at]);
      y[r] += A.val[at] * x[A.col[at]];
    }
  }
  for (size_t k = 0; k < A.long_row.size(); ++k)
    for (int64_t q = A.long_ptr[k]; q < A.long_ptr[k + 1]; ++q) y[A.long_row[k]] += A.long_val[q] * x[A.long_col[q]];
  f = fopen(argv[5], "wb");
  if (!f || fwrite(y.data(), 8, n, f) != (size_t)n) return fail("write");
  fclose(f);
  printf("OK %g %d\n", windows, (int)fits);
  return 0;
}
