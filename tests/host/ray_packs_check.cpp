// Test harness (CPU only): the sliced layout that appga_matrix_create builds of
// A (ray_packs, zorder, build_sell) of a CSR read from a binary file, for every
// number of lanes, unpacked and compared with the CSR.
//
//   ray_packs_check <in.bin>
//
// in.bin: int32 n, n_angles, m, nnz; int32 row_ptr[m+1]; int32 col[nnz]; float
// val[nnz].  Prints, per number of lanes: lanes, build_sell's result, rows that
// differ from the CSR's (as multisets of entries).
#include <algorithm>
#include <cstdio>
#include <string>
#include <utility>
#include <vector>

#include "appga_internal.h"

int main(int argc, char** argv) {
  if (argc != 2) return 2;
  FILE* in = std::fopen(argv[1], "rb");
  int32_t h[4];
  if (!in || std::fread(h, 4, 4, in) != 4) return 3;
  const int32_t n = h[0], na = h[1], m = h[2], nnz = h[3];
  std::vector<int32_t> ptr((size_t)m + 1), col((size_t)nnz);
  std::vector<float> val((size_t)nnz);
  if (std::fread(ptr.data(), 4, ptr.size(), in) != ptr.size() ||
      std::fread(col.data(), 4, col.size(), in) != col.size() ||
      std::fread(val.data(), 4, val.size(), in) != val.size())
    return 4;
  std::fclose(in);
  appga::HostCSR pl;
  appga::ray_packs(m, n, ptr.data(), col.data(), val.data(), &pl);
  for (int lanes : {1, 2, 4, 8}) {
    const int rows = 32 / lanes;
    std::vector<int32_t> order = appga::zorder(na, m / na);
    order.resize(((size_t)m + rows - 1) / rows * rows, -1);
    appga::HostSell s;
    const bool ok = appga::build_sell(order, lanes, pl.row_ptr, pl.col, pl.val, &s);
    int wrong = 0;
    for (size_t at = 0; ok && at < order.size(); ++at) {
      // the row's lanes of its slice: 20 bits of base column, three 14-bit offsets
      std::vector<std::pair<int32_t, float>> got, want;
      const int32_t slice = (int32_t)at / rows, lane0 = (int32_t)at % rows * lanes;
      for (int32_t p = s.off[slice]; p < s.off[slice + 1]; p += 32)
        for (int l = lane0; l < lane0 + lanes; ++l) {
          const uint64_t w = s.cols[(size_t)p + l];
          const int32_t base = (int32_t)(w & 0xfffff);
          for (int u = 0; u < 4; ++u) {
            int32_t d = u == 0 ? 0 : (int32_t)(w >> (20 + 14 * (u - 1)) & 0x3fff);
            if (d >= 8192) d -= 16384;
            const float v = s.vals[4 * ((size_t)p + l) + u];
            if (v != 0.f) got.emplace_back(base + d, v);
          }
        }
      const int32_t r = order[at];
      for (int32_t p = r < 0 ? 0 : ptr[r]; p < (r < 0 ? 0 : ptr[r + 1]); ++p)
        if (val[p] != 0.f)
          want.emplace_back(appga::tiled_index(col[p] / n, col[p] % n, n), val[p]);
      std::sort(got.begin(), got.end());
      std::sort(want.begin(), want.end());
      wrong += got != want;
    }
    std::printf("%d %d %d\n", lanes, ok ? 1 : 0, wrong);
  }
  return 0;
}
