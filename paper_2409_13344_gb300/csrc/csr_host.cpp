// Host-side CSR utilities: validation, stable transpose, row padding and the
// FP32 -> BF16 rounding of A's values.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <string>
#include <system_error>
#include <thread>
#include <tuple>
#include <utility>

#include "appga_internal.h"

namespace appga {

namespace {
// Parts that a pass over `entries` entries is worth splitting into, a thread each
// (starting one costs what some 2^16 entries do).
int host_parts(int64_t entries) {
  const int64_t cores = std::min(16u, std::max(1u, std::thread::hardware_concurrency()));
  return (int)std::max<int64_t>(1, std::min(cores, entries >> 17));
}
// body(first, last, part) over the parts of [0, n), which must not throw; a part
// whose thread cannot be had runs here.
template <class F>
void in_parts(int32_t n, int parts, F body) {
  std::vector<std::thread> threads;
  threads.reserve((size_t)parts);
  auto at = [&](int p) { return (int32_t)((int64_t)n * p / parts); };
  for (int p = 1; p < parts; ++p) {
    try {
      threads.emplace_back(body, at(p), at(p + 1), p);
    } catch (const std::system_error&) {
      body(at(p), at(p + 1), p);
    }
  }
  body(at(0), at(1), 0);
  for (auto& t : threads) t.join();
}
// Padded row starts: rows of a whole number of `mult` entries.
std::vector<int32_t> padded_starts(int32_t rows, const int32_t* row_ptr, int mult) {
  std::vector<int32_t> out((size_t)rows + 1, 0);
  for (int32_t i = 0; i < rows; ++i)
    out[(size_t)i + 1] = out[(size_t)i] + (row_ptr[i + 1] - row_ptr[i] + mult - 1) / mult * mult;
  return out;
}
}  // namespace

appga_status validate_csr(int32_t m, int32_t d, const int32_t* row_ptr, const int32_t* col,
                          const float* val, std::string* why) {
  if (m < 0 || d <= 0) {
    *why = "matrix shape must have m >= 0 and d > 0";
    return APPGA_EINVAL;
  }
  if (row_ptr == nullptr) {
    *why = "row_ptr is NULL";
    return APPGA_EINVAL;
  }
  if (row_ptr[0] != 0) {
    *why = "row_ptr[0] must be 0";
    return APPGA_EINVAL;
  }
  for (int32_t i = 0; i < m; ++i) {
    if (row_ptr[i + 1] < row_ptr[i]) {
      *why = "row_ptr must be nondecreasing (row " + std::to_string(i) + ")";
      return APPGA_EINVAL;
    }
  }
  const int64_t nnz = row_ptr[m];
  if (nnz > 0 && (col == nullptr || val == nullptr)) {
    *why = "col or val is NULL";
    return APPGA_EINVAL;
  }
  for (int64_t p = 0; p < nnz; ++p) {
    if (col[p] < 0 || col[p] >= d) {
      *why = "column index out of range at entry " + std::to_string(p);
      return APPGA_EINVAL;
    }
    const float v = val[p];
    if (!std::isfinite(v) || v < 0.f) {
      *why = "A must have finite nonnegative entries (entry " + std::to_string(p) + ")";
      return APPGA_EDOMAIN;
    }
  }
  return APPGA_OK;
}

void transpose_csr(int32_t m, int32_t d, const int32_t* row_ptr, const int32_t* col,
                   const float* val, HostCSR* out) {
  const int64_t nnz = row_ptr[m];
  out->rows = d;
  out->cols = m;
  out->row_ptr.assign((size_t)d + 1, 0);
  out->col.resize((size_t)nnz);
  out->val.resize((size_t)nnz);
  for (int64_t p = 0; p < nnz; ++p) out->row_ptr[(size_t)col[p] + 1]++;
  for (int32_t j = 0; j < d; ++j) out->row_ptr[j + 1] += out->row_ptr[j];
  std::vector<int32_t> next(out->row_ptr.begin(), out->row_ptr.end() - 1);
  // rows visited in order -> each transposed row lists ray indices ascending
  for (int32_t i = 0; i < m; ++i) {
    for (int32_t p = row_ptr[i]; p < row_ptr[i + 1]; ++p) {
      const int32_t q = next[col[p]]++;
      out->col[q] = i;
      out->val[q] = val[p];
    }
  }
}

void pad_rows(int32_t rows, int32_t cols, const int32_t* row_ptr, const int32_t* col,
              const float* val, int mult, HostCSR* out) {
  out->rows = rows;
  out->cols = cols;
  out->row_ptr = padded_starts(rows, row_ptr, mult);
  out->col.assign((size_t)out->row_ptr[rows], 0);
  out->val.assign((size_t)out->row_ptr[rows], 0.f);
  in_parts(rows, host_parts(row_ptr[rows]), [=](int32_t first, int32_t end, int) {
    for (int32_t i = first; i < end; ++i) {
      const int32_t s = row_ptr[i], e = row_ptr[i + 1];
      int32_t q = out->row_ptr[i];
      for (int32_t p = s; p < e; ++p, ++q) {
        out->col[q] = col[p];
        out->val[q] = val[p];
      }
      const int32_t last = e > s ? col[e - 1] : 0;
      for (; q < out->row_ptr[i + 1]; ++q) {
        out->col[q] = last;  // same cache line as the row's last gather
        out->val[q] = 0.f;
      }
    }
  });
}

bool encode_pack(const int32_t* c, uint64_t* word) {
  if (c[0] < 0 || c[0] > PACK_BASE_MAX) return false;
  uint64_t w = (uint64_t)c[0];
  for (int i = 1; i < PACK_ENTRIES; ++i) {
    const int32_t dlt = c[i] - c[0];
    if (dlt < -PACK_OFFSET_MAX - 1 || dlt > PACK_OFFSET_MAX) return false;
    w |= ((uint64_t)(uint32_t)dlt & 0x3fffull) << (PACK_BASE_BITS + 14 * (i - 1));
  }
  *word = w;
  return true;
}

bool pack_columns(const std::vector<int32_t>& col, std::vector<uint64_t>* out) {
  out->clear();
  if (col.size() % PACK_ENTRIES != 0) return false;
  const size_t np = col.size() / PACK_ENTRIES;
  out->resize(np);
  for (size_t q = 0; q < np; ++q)
    if (!encode_pack(&col[q * PACK_ENTRIES], &(*out)[q])) return false;
  return true;
}

bool build_sell(const std::vector<int32_t>& order, int lanes, const std::vector<int32_t>& row_ptr,
                const std::vector<int32_t>& col, const std::vector<float>& val, HostSell* out) {
  const int C = 32 / lanes, L = lanes;
  const int32_t ns = (int32_t)(order.size() / C);
  out->rows = (int32_t)order.size();
  out->slices = ns;
  out->lanes = L;
  out->off.assign((size_t)ns + 1, 0);
  auto packs = [&](int32_t r) { return r < 0 ? 0 : (row_ptr[r + 1] - row_ptr[r]) / PACK_ENTRIES; };
  // steps of a slice: the most packs of any of its rows, over the L lanes of a row
  int64_t total = 0;
  for (int32_t s = 0; s < ns; ++s) {
    int32_t most = 0;
    for (int q = 0; q < C; ++q) most = std::max(most, packs(order[(size_t)s * C + q]));
    const int64_t steps = (most + L - 1) / L;
    total += steps * 32;
    if (total > (int64_t)INT32_MAX) return false;
    out->off[(size_t)s + 1] = (int32_t)total;
  }
  out->cols.assign((size_t)total, 0ull);
  out->vals.assign((size_t)total * PACK_ENTRIES, 0.f);
  std::atomic<bool> fits{true};
  in_parts(ns, host_parts(total * PACK_ENTRIES), [&](int32_t first, int32_t end, int) {
    for (int32_t s = first; s < end && fits.load(std::memory_order_relaxed); ++s) {
      const int64_t base = out->off[(size_t)s];
      for (int q = 0; q < C; ++q) {
        const int32_t r = order[(size_t)s * C + q], npk = packs(r);
        // what is left of a row repeats a column of its last pack with zero
        // values: no vector entry that the row does not meet is read for it
        const int32_t steps = (out->off[(size_t)s + 1] - out->off[(size_t)s]) / 32;
        for (int32_t k = npk; npk > 0 && k < steps * L; ++k)
          out->cols[(size_t)(base + (int64_t)(k / L) * 32 + q * L + k % L)] =
              (uint64_t)col[(size_t)row_ptr[r + 1] - PACK_ENTRIES];
        for (int32_t k = 0; k < npk; ++k) {
          const int64_t pos = base + (int64_t)(k / L) * 32 + q * L + (k % L);
          const int32_t e = row_ptr[r] + k * PACK_ENTRIES;
          if (!encode_pack(&col[(size_t)e], &out->cols[(size_t)pos])) fits = false;
          for (int i = 0; i < PACK_ENTRIES; ++i)
            out->vals[(size_t)pos * PACK_ENTRIES + i] = val[(size_t)e + i];
        }
      }
    }
  });
  return fits;
}

bool build_sell(int32_t rows, const std::vector<int32_t>& row_ptr, const std::vector<int32_t>& col,
                const std::vector<float>& val, HostSell* out) {
  std::vector<int32_t> order(((size_t)rows + 7) / 8 * 8, -1);
  for (int32_t r = 0; r < rows; ++r) order[(size_t)r] = r;
  if (!build_sell(order, 4, row_ptr, col, val, out)) return false;
  out->rows = rows;
  return true;
}

void ray_packs(int32_t rows, int32_t n, const int32_t* row_ptr, const int32_t* col,
               const float* val, HostCSR* out) {
  out->rows = rows;
  out->cols = n * n;
  out->row_ptr = padded_starts(rows, row_ptr, PACK_ENTRIES);
  out->col.assign((size_t)out->row_ptr[rows], 0);
  out->val.assign((size_t)out->row_ptr[rows], 0.f);
  int32_t longest = 0;
  for (int32_t i = 0; i < rows; ++i) longest = std::max(longest, row_ptr[i + 1] - row_ptr[i]);
  const int parts = host_parts(row_ptr[rows]);
  // per part, for the row at hand: the pixel (row, column) of each entry, the
  // entries in ray order, and the entries that start each column
  struct Scratch {
    std::vector<std::pair<int32_t, int32_t>> at;
    std::vector<int32_t> order, start;
  };
  std::vector<Scratch> scratch((size_t)parts);
  for (auto& x : scratch) {
    x.at.resize((size_t)longest);
    x.order.resize((size_t)longest);
    x.start.resize((size_t)n + 1);
  }
  in_parts(rows, parts, [&](int32_t first, int32_t end, int part) {
    auto* at = scratch[(size_t)part].at.data();
    int32_t* order = scratch[(size_t)part].order.data();
    int32_t* start = scratch[(size_t)part].start.data();
    for (int32_t i = first; i < end; ++i) {
      const int32_t s = row_ptr[i], len = row_ptr[i + 1] - s;
      if (len == 0) continue;
      int32_t c0 = n, c1 = -1, r0 = n, r1 = -1;
      bool ascending = true;
      for (int32_t k = 0; k < len; ++k) {
        const int32_t r = col[s + k] / n, c = col[s + k] - r * n;
        at[k] = {r, c};
        r0 = std::min(r0, r);
        r1 = std::max(r1, r);
        c0 = std::min(c0, c);
        c1 = std::max(c1, c);
        order[k] = k;
        ascending &= k == 0 || col[s + k] >= col[s + k - 1];
      }
      if (c1 - c0 > r1 - r0) {  // by column (ascending indices are by row already)
        if (ascending) {        // a stable counting sort
          std::fill(start + c0, start + c1 + 1, 0);
          for (int32_t k = 0; k < len; ++k) ++start[at[k].second];
          for (int32_t c = c0, sum = 0; c <= c1; ++c) {
            const int32_t count = start[c];
            start[c] = sum;
            sum += count;
          }
          for (int32_t k = 0; k < len; ++k) order[start[at[k].second]++] = k;
        } else {
          std::sort(order, order + len, [at](int32_t a, int32_t b) {
            return std::make_tuple(at[a].second, at[a].first, a) <
                   std::make_tuple(at[b].second, at[b].first, b);
          });
        }
      }
      int32_t* pc = &out->col[(size_t)out->row_ptr[i]];
      float* pv = &out->val[(size_t)out->row_ptr[i]];
      const int32_t padded = out->row_ptr[i + 1] - out->row_ptr[i];
      auto place = [&] {
        for (int32_t k = 0; k < len; ++k) {
          pc[k] = tiled_index(at[order[k]].first, at[order[k]].second, n);
          pv[k] = val[s + order[k]];
        }
        for (int32_t k = len; k < padded; ++k) pc[k] = pc[len - 1];
      };
      place();
      // a row that covers a wide strip steps too far from one column to the next
      bool fits = true;
      uint64_t word;
      for (int32_t k = 0; fits && k < padded; k += PACK_ENTRIES) fits = encode_pack(pc + k, &word);
      if (!fits) {
        for (int32_t k = 0; k < len; ++k) order[k] = k;
        place();
      }
    }
  });
}

bool quarter_turn_symmetric(int32_t m, int32_t n, int32_t n_angles, const int32_t* row_ptr,
                            const int32_t* col, const float* val) {
  if (n < 2 || n % 2 != 0 || n_angles < 2 || n_angles % 2 != 0 || m % n_angles != 0)
    return false;
  const int32_t nb = m / n_angles, half = m / 2, d = n * n;
  // pos[c] (of a part): entry of the partner row at column c (-1 none); an entry
  // matched by a turned column of row i is marked -2, so a repeat fails
  const int parts = host_parts(row_ptr[half]);
  std::vector<std::vector<int32_t>> seen((size_t)parts, std::vector<int32_t>((size_t)d, -1));
  std::atomic<bool> same{true};
  in_parts(half, parts, [&](int32_t first, int32_t end, int part) {
    int32_t* pos = seen[(size_t)part].data();
    for (int32_t i = first; i < end && same.load(std::memory_order_relaxed); ++i) {
      const int32_t k = fold_partner(i, half, nb);
      bool ok = row_ptr[k + 1] - row_ptr[k] == row_ptr[i + 1] - row_ptr[i];
      int32_t p = row_ptr[k];
      for (; ok && p < row_ptr[k + 1]; ++p) {
        if (pos[col[p]] != -1) {
          ok = false;
          break;
        }
        pos[col[p]] = p;
      }
      for (int32_t q = row_ptr[i]; ok && q < row_ptr[i + 1]; ++q) {
        const int32_t t = quarter_turn(col[q], n);
        const int32_t at = pos[t];
        ok = at >= 0 && std::memcmp(&val[at], &val[q], sizeof(float)) == 0;
        if (ok) pos[t] = -2;
      }
      for (int32_t r = row_ptr[k]; r < p; ++r) pos[col[r]] = -1;
      if (!ok) same = false;
    }
  });
  return same;
}

void fold_transpose(const HostCSR& at, int32_t half, int32_t n, HostCSR* out) {
  const int32_t d = at.rows;
  out->rows = d;
  out->cols = half;
  out->row_ptr.assign((size_t)d + 1, 0);
  auto pixel = [n](int32_t k) {
    int32_t r, c;
    orbit_pixel(k / 4, k % 4, n, &r, &c);
    return r * n + c;
  };
  // rows of at list ray indices ascending: the first half is a prefix
  for (int32_t k = 0; k < d; ++k) {
    const int32_t p = pixel(k);
    const auto row = at.col.begin() + at.row_ptr[p], end = at.col.begin() + at.row_ptr[p + 1];
    out->row_ptr[(size_t)k + 1] =
        out->row_ptr[(size_t)k] + (int32_t)(std::lower_bound(row, end, half) - row);
  }
  out->col.resize((size_t)out->row_ptr[d]);
  out->val.resize((size_t)out->row_ptr[d]);
  in_parts(d, host_parts(out->row_ptr[d]), [&](int32_t first, int32_t last, int) {
    for (int32_t k = first; k < last; ++k) {
      const int32_t from = at.row_ptr[pixel(k)], len = out->row_ptr[k + 1] - out->row_ptr[k];
      if (len == 0) continue;
      std::copy_n(&at.col[from], len, &out->col[out->row_ptr[k]]);
      std::copy_n(&at.val[from], len, &out->val[out->row_ptr[k]]);
    }
  });
}

void tile_columns(int32_t n, std::vector<int32_t>* col) {
  const int32_t size = (int32_t)col->size();
  in_parts(size, host_parts(size), [=](int32_t first, int32_t end, int) {
    for (int32_t q = first; q < end; ++q) {
      const int32_t j = (*col)[(size_t)q];
      (*col)[(size_t)q] = tiled_index(j / n, j % n, n);
    }
  });
}

std::vector<int32_t> zorder(int32_t ny, int32_t nx) {
  std::vector<int32_t> out;
  out.reserve((size_t)ny * nx);
  int64_t side = 1;
  while (side < ny || side < nx) side *= 2;
  // squares of the curve that still meet the grid, as (y, x, side) on a stack
  struct Square {
    int64_t y, x, side;
  };
  std::vector<Square> todo = {{0, 0, side}};
  while (!todo.empty()) {
    const Square q = todo.back();
    todo.pop_back();
    if (q.y >= ny || q.x >= nx) continue;
    if (q.side == 1) {
      out.push_back((int32_t)(q.y * nx + q.x));
      continue;
    }
    const int64_t h = q.side / 2;
    todo.push_back({q.y + h, q.x + h, h});
    todo.push_back({q.y + h, q.x, h});
    todo.push_back({q.y, q.x + h, h});
    todo.push_back({q.y, q.x, h});
  }
  return out;
}

uint16_t float_to_bf16(float x) {
  uint32_t u;
  std::memcpy(&u, &x, 4);
  if ((u & 0x7f800000u) == 0x7f800000u) return (uint16_t)(u >> 16);  // inf / nan (not expected)
  const uint32_t lsb = (u >> 16) & 1u;
  u += 0x7fffu + lsb;  // round to nearest, ties to even
  return (uint16_t)(u >> 16);
}

}  // namespace appga
