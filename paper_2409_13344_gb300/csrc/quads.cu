// Row-block layout of the batched projectors' matrices, built on the device
// from the row-padded CSR.
//
// Four rows that are neighbours in the row order (a 2 x 2 tile of pixels, or
// rays of two bins and two angles) share most of the columns they meet.  A
// block keeps their union of columns, each with its four values (zero where a
// row does not meet it), so a gathered row of the slot-minor vector serves up
// to four rows from registers: on a parallel-beam matrix a union column serves
// 2.0 pixels, or 1.5 rays.
#include <cuda_runtime.h>

#include <vector>

#include "appga_internal.h"
#include "handles.h"

namespace appga {
namespace {

// The merge of a block's four rows, one union column at a time.  Rows need not
// be sorted: every entry is taken exactly once, with its own column.  Zero
// entries (the rows' padding) are left out.
struct Merge {
  int p[4], e[4];
  __device__ Merge(const DevCSR& M, int b) {
    for (int r = 0; r < 4; ++r) {
      const int q = 4 * b + r;
      const int row = q < M.rows ? (M.order ? M.order[q] : q) : -1;
      p[r] = row >= 0 ? M.row_ptr[row] : 0;
      e[r] = row >= 0 ? M.row_ptr[row + 1] : 0;
    }
  }
  // the next union column and the entry of each row there (-1: none); false
  // at the end
  __device__ bool next(const DevCSR& M, int& col, int (&at)[4]) {
    int c[4];
    col = 0x7fffffff;
    for (int r = 0; r < 4; ++r) {
      while (p[r] < e[r] && M.val[p[r]] == 0.f) ++p[r];
      c[r] = p[r] < e[r] ? M.col[p[r]] : 0x7fffffff;
      col = min(col, c[r]);
    }
    if (col == 0x7fffffff) return false;
    for (int r = 0; r < 4; ++r) {
      at[r] = c[r] == col ? p[r] : -1;
      if (at[r] >= 0) ++p[r];
    }
    return true;
  }
};

__global__ void k_quad_count(DevCSR M, int blocks, int* __restrict__ packs) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= blocks) return;
  Merge m(M, b);
  int col, at[4], n = 0;
  while (m.next(M, col, at)) ++n;
  packs[b] = (n + 3) / 4;
}

__global__ void k_quad_fill(DevCSR M, DevQuad Q) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= Q.blocks) return;
  for (int r = 0; r < 4; ++r) {
    const int q = 4 * b + r;
    Q.rows[q] = q < M.rows ? (M.order ? M.order[q] : q) : -1;
  }
  Merge m(M, b);
  int col = 0, at[4];
  bool more = true;
  for (int k = Q.off[b]; k < Q.off[b + 1]; ++k) {
    int c[4];
    for (int u = 0; u < 4; ++u) {
      const int last = col;
      if (more) more = m.next(M, col, at);
      if (!more) col = last;  // padding: the last column again, with zeros
      c[u] = col;
      float v[4];
      uint16_t h[4];
      for (int r = 0; r < 4; ++r) {
        const bool have = more && at[r] >= 0;
        v[r] = have ? M.val[at[r]] : 0.f;
        h[r] = have && M.val_bf16 ? M.val_bf16[at[r]] : (uint16_t)0;
      }
      const size_t o = (size_t)4 * k + u;
      Q.vals[o] = make_float4(v[0], v[1], v[2], v[3]);
      if (Q.vals_bf16)
        Q.vals_bf16[o] = make_uint2(h[0] | (uint32_t)h[1] << 16, h[2] | (uint32_t)h[3] << 16);
    }
    Q.cols[k] = make_int4(c[0], c[1], c[2], c[3]);
  }
}

appga_status build(const DevCSR& M, cudaStream_t s, DevQuad* out, int64_t* bytes) {
  DevQuad q;
  q.blocks = (M.rows + 3) / 4;
  std::vector<int32_t> off((size_t)q.blocks + 1);
  cudaError_t e = dalloc(&q.off, (size_t)q.blocks + 1, bytes);
  if (e == cudaSuccess) e = dalloc(&q.rows, (size_t)4 * q.blocks, bytes);
  const int grid = (q.blocks + 63) / 64;
  if (e == cudaSuccess) {
    k_quad_count<<<grid, 64, 0, s>>>(M, q.blocks, q.off + 1);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(off.data() + 1, q.off + 1, (size_t)q.blocks * 4, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e == cudaSuccess) {
    off[0] = 0;
    for (int b = 0; b < q.blocks; ++b) off[b + 1] += off[b];  // packs <= entries / 2: fits
    const size_t np = (size_t)off[q.blocks];
    e = cudaMemcpyAsync(q.off, off.data(), off.size() * 4, cudaMemcpyHostToDevice, s);
    // (the projectors' L2 prefetches run up to 64 packs past the end)
    if (e == cudaSuccess) e = dalloc(&q.cols, np + 64, bytes);
    if (e == cudaSuccess) e = dalloc(&q.vals, 4 * np + 256, bytes);
    if (e == cudaSuccess && M.val_bf16) e = dalloc(&q.vals_bf16, 4 * np + 256, bytes);
  }
  if (e == cudaSuccess) {
    k_quad_fill<<<grid, 64, 0, s>>>(M, q);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    free_quad(q);
    return cuda_fail(e, "batched matrix layout");
  }
  *out = q;
  return APPGA_OK;
}

}  // namespace

void free_quad(DevQuad& q) {
  cudaFree(q.off);
  cudaFree(q.rows);
  cudaFree(q.cols);
  cudaFree(q.vals);
  cudaFree(q.vals_bf16);
  q = DevQuad();
}

appga_status ensure_quads(appga_matrix* M, cudaStream_t s) {
  if (M->quad_a.off == nullptr) {
    const appga_status rc = build(M->A, s, &M->quad_a, &M->bytes);
    if (rc != APPGA_OK) return rc;
  }
  if (M->quad_t.off == nullptr) return build(M->At, s, &M->quad_t, &M->bytes);
  return APPGA_OK;
}

}  // namespace appga
