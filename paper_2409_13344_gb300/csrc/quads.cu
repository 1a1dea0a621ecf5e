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

// The merge of a block's four rows by four lanes, a row each, one union column
// at a time.  Rows need not be sorted: every entry is taken exactly once, with
// its own column.  Zero entries (the rows' padding) are left out.  What bounds
// it is the chain of steps, so a lane holds the 4-entry pack of its head and the
// pack after it, and a step waits for no load.  With one thread per block, which
// walked the four rows through memory, the first batched call of a matrix took
// 2.2 ms at 64 x 64 (48 angles), 11.5 at 256 x 256 (180) and 34.4 at 512 x 512
// (360) for 20 maps of 5 slices; 1.6, 6.2 and 25.8 so (0.55, 3.0 and 16.9 ms of
// them the call itself).
struct Merge {
  const int32_t* col;
  const float* val;
  int p, e;       // the head's entry and the row's end (a multiple of 4, as every row start)
  int4 c, cn;     // columns of the head's pack and of the next
  float4 v, vn;
  __device__ Merge(const DevCSR& M, int b, int r) : col(M.col), val(M.val) {
    const int q = 4 * b + r;
    const int row = q < M.rows ? (M.order ? M.order[q] : q) : -1;
    p = row >= 0 ? M.row_ptr[row] : 0;
    e = row >= 0 ? M.row_ptr[row + 1] : 0;
    c = cn = make_int4(0, 0, 0, 0);
    v = vn = make_float4(0.f, 0.f, 0.f, 0.f);
    if (p < e) fetch(p, c, v);
    if (p + 4 < e) fetch(p + 4, cn, vn);
    skip();
  }
  __device__ void fetch(int at, int4& cc, float4& vv) const {
    cc = *reinterpret_cast<const int4*>(col + at);
    vv = *reinterpret_cast<const float4*>(val + at);
  }
  __device__ int head() const {
    if (p >= e) return 0x7fffffff;
    return p & 2 ? (p & 1 ? c.w : c.z) : (p & 1 ? c.y : c.x);
  }
  __device__ float value() const { return p & 2 ? (p & 1 ? v.w : v.z) : (p & 1 ? v.y : v.x); }
  __device__ void step() {
    if ((++p & 3) == 0) {
      c = cn;
      v = vn;
      if (p + 4 < e) fetch(p + 4, cn, vn);
    }
  }
  __device__ void skip() {
    while (p < e && value() == 0.f) step();
  }
  // the next union column, in the block's four lanes, and this lane's entry
  // there (-1: none); false at the end
  __device__ bool next(int& column, int& at) {
    const int h = head();
    int m = min(h, __shfl_xor_sync(0xffffffffu, h, 1));
    m = min(m, __shfl_xor_sync(0xffffffffu, m, 2));
    if (m == 0x7fffffff) return false;
    column = m;
    at = h == m ? p : -1;
    return true;
  }
  __device__ void take(int at) {
    if (at < 0) return;
    step();
    skip();
  }
};

// (a warp works until the longest of its eight blocks is done)
__global__ void __launch_bounds__(128) k_quad_count(DevCSR M, int blocks, int* __restrict__ packs) {
  const int b = (blockIdx.x * blockDim.x + threadIdx.x) / 4, r = threadIdx.x & 3;
  Merge m(M, b, r);
  int col, at, n = 0;
  bool more = true;
  while (__any_sync(0xffffffffu, more)) {
    more = m.next(col, at);
    if (more) {
      ++n;
      m.take(at);
    }
  }
  if (r == 0 && b < blocks) packs[b] = (n + 3) / 4;
}

__global__ void __launch_bounds__(128) k_quad_fill(DevCSR M, DevQuad Q) {
  const int b = (blockIdx.x * blockDim.x + threadIdx.x) / 4, r = threadIdx.x & 3;
  if (b < Q.blocks) {
    const int q = 4 * b + r;
    Q.rows[q] = q < M.rows ? (M.order ? M.order[q] : q) : -1;
  }
  Merge m(M, b, r);
  // union column o of the layout: its column, and its four values by the lanes
  size_t o = b < Q.blocks ? (size_t)4 * Q.off[b] : 0;
  const size_t end = b < Q.blocks ? (size_t)4 * Q.off[b + 1] : 0;
  int col = 0, at = -1;
  bool more = true;
  while (__any_sync(0xffffffffu, more || o < end)) {
    more = m.next(col, at);
    if (o < end) {  // past the last union column: that column again, with zeros
      const bool have = more && at >= 0;
      if (r == 0) reinterpret_cast<int32_t*>(Q.cols)[o] = col;
      reinterpret_cast<float*>(Q.vals)[4 * o + r] = have ? m.value() : 0.f;
      if (Q.vals_bf16)
        reinterpret_cast<uint16_t*>(Q.vals_bf16)[4 * o + r] =
            have && M.val_bf16 ? M.val_bf16[at] : (uint16_t)0;
      ++o;
    }
    if (more) m.take(at);
  }
}

// 32 blocks of rows per thread block
int grid_of(const DevQuad& q) { return (q.blocks + 31) / 32; }

// The blocks of M: their rows' places and the packs of each, without the packs.
appga_status count(const DevCSR& M, cudaStream_t s, DevQuad* out, int64_t* bytes) {
  DevQuad q;
  int64_t held = 0;
  q.blocks = (M.rows + 3) / 4;
  std::vector<int32_t> off((size_t)q.blocks + 1);
  cudaError_t e = dalloc(&q.off, (size_t)q.blocks + 1, &held);
  if (e == cudaSuccess) e = dalloc(&q.rows, (size_t)4 * q.blocks, &held);
  if (e == cudaSuccess) {
    k_quad_count<<<grid_of(q), 128, 0, s>>>(M, q.blocks, q.off + 1);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(off.data() + 1, q.off + 1, (size_t)q.blocks * 4, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e == cudaSuccess) {
    off[0] = 0;
    for (int b = 0; b < q.blocks; ++b) off[b + 1] += off[b];  // packs <= entries / 2: fits
    q.packs = off[q.blocks];
    e = cudaMemcpyAsync(q.off, off.data(), off.size() * 4, cudaMemcpyHostToDevice, s);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    free_quad(q);
    return cuda_fail(e, "batched matrix layout");
  }
  *out = q;
  *bytes += held;
  return APPGA_OK;
}

// Packs allocated (the projectors' L2 prefetches run up to 64 past the end).
size_t packs_held(const DevQuad& q) { return (size_t)q.packs + 64; }

appga_status fill(const DevCSR& M, cudaStream_t s, DevQuad* out, int64_t* bytes) {
  DevQuad q = *out;
  int64_t held = 0;
  cudaError_t e = dalloc(&q.cols, packs_held(q), &held);
  if (e == cudaSuccess) e = dalloc(&q.vals, 4 * packs_held(q), &held);
  if (e == cudaSuccess && M.val_bf16) e = dalloc(&q.vals_bf16, 4 * packs_held(q), &held);
  if (e == cudaSuccess) {
    k_quad_fill<<<grid_of(q), 128, 0, s>>>(M, q);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    cudaFree(q.cols);
    cudaFree(q.vals);
    cudaFree(q.vals_bf16);
    return cuda_fail(e, "batched matrix layout");
  }
  *out = q;
  *bytes += held;
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

namespace {
appga_status ensure_counts(appga_matrix* M, cudaStream_t s) {
  appga_status rc = APPGA_OK;
  if (M->quad_a.off == nullptr) rc = count(M->A, s, &M->quad_a, &M->bytes);
  if (rc == APPGA_OK && M->quad_t.off == nullptr) rc = count(M->At, s, &M->quad_t, &M->bytes);
  return rc;
}
}  // namespace

appga_status quad_bytes_missing(appga_matrix* M, cudaStream_t s, int64_t* bytes) {
  const appga_status rc = ensure_counts(M, s);
  if (rc != APPGA_OK) return rc;
  *bytes = 0;
  const int64_t pack = sizeof(int4) + 4 * (sizeof(float4) + (M->A.val_bf16 ? sizeof(uint2) : 0));
  if (M->quad_a.cols == nullptr) *bytes += (int64_t)packs_held(M->quad_a) * pack;
  if (M->quad_t.cols == nullptr) *bytes += (int64_t)packs_held(M->quad_t) * pack;
  return APPGA_OK;
}

appga_status ensure_quads(appga_matrix* M, cudaStream_t s) {
  appga_status rc = ensure_counts(M, s);
  if (rc == APPGA_OK && M->quad_a.cols == nullptr) rc = fill(M->A, s, &M->quad_a, &M->bytes);
  if (rc == APPGA_OK && M->quad_t.cols == nullptr) rc = fill(M->At, s, &M->quad_t, &M->bytes);
  return rc;
}

}  // namespace appga
