// Batched CUDA kernels: K independent slices (slots) that share one system
// matrix run the APPGA iteration together, so every nonzero of A and A^T is
// read once per iteration for all K right-hand sides (CSR SpMM).
//
// Layout (slot-minor): images f[j][s], sinograms y[i][s], w[i][s], g[i][s],
// rows of Kp slots.  A launch works on the first W = 8, 16, 32, 64 or 128 of
// them; the lanes of a warp share a row's products as Team<W> says.  The bound
// is the L1 pipe: each nonzero takes W/32 passes of 128 bytes for its gathered
// row, plus its share of the matrix's broadcast loads.  Rows are dealt to
// warps along a Z-order curve (pixels, or rays by angle and bin), so a block
// gathers for neighbouring rows and half to three quarters of the sectors hit
// L1 (64 slots of 256 x 256: 1.8 and 1.2 GB from L2 per projection, 3.5 and
// 2.6 GB in row order).  The per-(row, slot) epilogues match the single-slice
// kernels (Eq. APPGAiter, Eq. EM, Sec. 2.2); the SHOITV stencil is a kernel of
// its own that runs beside the forward projection.
//
// Every slot carries its own device state (iteration index, momentum scalar,
// objective, stop flag, parameters), so slots may sit at different
// iterations (continuous batching).  The iterate rings are indexed by a
// global step counter shared by all slots.  Per-slot objective sums use the
// deterministic two-level grid reduction, so results do not depend on which
// other slots are in the batch.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "appga_internal.h"
#include "batched_internal.h"
#include "device_common.cuh"

namespace appga {
namespace {

constexpr int B_THREADS = 256;               // stencil blocks (and set-up kernels)
constexpr int MAXK = 128;                    // largest padded batch
// Projector blocks: 16 warps, two blocks per SM (64 registers per thread).  A
// block's warps work on a compact bundle of rows (DevCSR::order), so the wider
// the block the more of its gathers meet in L1.
constexpr int P_THREADS = 512;
constexpr int P_WARPS = P_THREADS / 32;
constexpr int kMaxPerSm = 16;                // upper bound of the tuned values
__host__ __forceinline__ int clamp_per_sm(int v, int dflt) {
  return v <= 0 ? dflt : (v > kMaxPerSm ? kMaxPerSm : v);
}
// Row groups per SM when no tuned schedule is given: more than are resident
// at once, so the block scheduler levels the tail.
constexpr int kSpmvPerSm = 8;
constexpr int kPixelPerSm = 8;
constexpr int kStencilPerSm = 8;
// Stencil blocks: 8 slots x 32 image columns (the outer two on each side are
// halo), marching down runs of BST_R rows.
constexpr int BST_S = 8, BST_C = B_THREADS / BST_S, BST_OUT = BST_C - 4, BST_R = 16;
static_assert(BST_S == 8 && BST_C % 4 == 0, "a warp holds four columns of eight slots");

template <int E>
__device__ __forceinline__ void vload(const float* p, float (&x)[E]) {
  if constexpr (E == 1) {
    x[0] = *p;
  } else if constexpr (E == 2) {
    const float2 t = *reinterpret_cast<const float2*>(p);
    x[0] = t.x;
    x[1] = t.y;
  } else {
    const float4 t = *reinterpret_cast<const float4*>(p);
    x[0] = t.x;
    x[1] = t.y;
    x[2] = t.z;
    x[3] = t.w;
  }
}
// Stores the elements whose on[] is set (one vector store when all are).
template <int E>
__device__ __forceinline__ void vstore_on(float* p, const float (&x)[E], const int (&on)[E]) {
  int all = 1;
#pragma unroll
  for (int t = 0; t < E; ++t) all &= on[t] ? 1 : 0;
  if (all) {
    if constexpr (E == 1) {
      *p = x[0];
    } else if constexpr (E == 2) {
      *reinterpret_cast<float2*>(p) = make_float2(x[0], x[1]);
    } else {
      *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
    }
  } else {
#pragma unroll
    for (int t = 0; t < E; ++t)
      if (on[t]) p[t] = x[t];
  }
}

// How the lanes of a warp share a row whose products fill W slots.  A lane
// holds Q slots (Q/4 16-byte loads per gathered row), L lanes make a group
// that covers the W slots, and the G groups of a row's team take the row's
// 4-entry packs in turn.  The row's sum is always that of four partial sums,
// p_i over the packs k = i (mod 4) in order, as (p0 + p1) + (p2 + p3), so the
// results do not depend on W: the widest team holds several of the four in
// one lane (A), the narrow ones work on RW rows of the warp at a time.
// Eight slots per lane because the load of a pack's columns or values, which
// a group's lanes make at one address, still takes the L1 pipe four passes
// (a 16-byte load is served in quarter warps): with four groups a warp those
// passes feed 16 entries.
template <int W>
struct Team {
  static constexpr int Q = W >= 16 ? 8 : 4;
  static constexpr int L = W / Q;
  static constexpr int G = L <= 8 ? 4 : 32 / L;
  static constexpr int A = 4 / G;
  static constexpr int LANES = L * G;
  static constexpr int RW = 32 / LANES;
  static constexpr int E = Q / G;  // slots a lane owns after the reduction
  static constexpr int GSTRIDE = 4 * L;
};
// A lane gathers the slots gathered_slot + i * GSTRIDE .. + 3, i < Q/4 (so
// that a quarter warp's 16-byte loads are consecutive: one pass each), and
// owns the E slots from owned_slot after the reduction.
template <int W>
__device__ __forceinline__ int gathered_slot(int lane) {
  return 4 * (lane % Team<W>::L);
}
template <int W>
__device__ __forceinline__ int owned_slot(int lane) {
  using T = Team<W>;
  const int g = lane % T::LANES / T::L;
  if constexpr (T::Q == 4) return gathered_slot<W>(lane) + 2 * (g & 1) + (g >> 1);
  return gathered_slot<W>(lane) + T::GSTRIDE * (g & 1) + T::E * (g >> 1);
}

// One row of M (row < 0: none) times the columns of X ([cols][stride]): each
// lane ends with the sums of the E slots from owned_slot.  A lane gathers NZ
// (2 or 4) entries of a pack per step while the columns and values of the
// next pack are in flight; `on`: some of the lane's gathered slots is wanted.
// All lanes of the warp take part.
template <int W, bool BF16, int NZ>
__device__ __forceinline__ void team_dot(const DevCSR& M, int row, const float* __restrict__ X,
                                         int stride, int lane, bool on, uint64_t pol,
                                         float (&out)[Team<W>::E]) {
  using T = Team<W>;
  constexpr int A = T::A, Q = T::Q, F = Q / 4, E = T::E;
  const int g = lane % T::LANES / T::L;
  int p = 0, cnt = 0;  // the lane's packs are g, g + G, ...: cnt of them from p
  if (row >= 0 && on) {
    const int s = __ldg(M.row_ptr + row);
    const int npk = (__ldg(M.row_ptr + row + 1) - s) >> 2;
    cnt = npk > g ? (npk - g + T::G - 1) / T::G : 0;
    p = s + 4 * g;
  }
  const float* xl = X + gathered_slot<W>(lane);
  float acc[A][Q];
#pragma unroll
  for (int i = 0; i < A; ++i)
#pragma unroll
    for (int q = 0; q < Q; ++q) acc[i][q] = 0.f;
  int4 c = make_int4(0, 0, 0, 0);
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (cnt > 0) {
    c = ld_stream_i4(M.col + p, pol);
    v = ld_vals<BF16>(M, p, pol);
  }
  auto pack = [&](float (&a)[Q], bool more) {
    const int cc[4] = {c.x, c.y, c.z, c.w};
    const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int h = 0; h < 4; h += NZ) {
      float4 x[NZ][F];
#pragma unroll
      for (int u = 0; u < NZ; ++u)
#pragma unroll
        for (int i = 0; i < F; ++i)
          x[u][i] = __ldg(reinterpret_cast<const float4*>(xl + (unsigned)(cc[h + u] * stride)) +
                          i * (T::GSTRIDE / 4));
      if (h + NZ == 4 && more) {
        p += 4 * T::G;
        c = ld_stream_i4(M.col + p, pol);
        v = ld_vals<BF16>(M, p, pol);
      }
#pragma unroll
      for (int u = 0; u < NZ; ++u)
#pragma unroll
        for (int i = 0; i < F; ++i) {
          a[4 * i] = fmaf(vv[h + u], x[u][i].x, a[4 * i]);
          a[4 * i + 1] = fmaf(vv[h + u], x[u][i].y, a[4 * i + 1]);
          a[4 * i + 2] = fmaf(vv[h + u], x[u][i].z, a[4 * i + 2]);
          a[4 * i + 3] = fmaf(vv[h + u], x[u][i].w, a[4 * i + 3]);
        }
    }
  };
  int j = 0;
  for (; j + A < cnt; j += A) {  // all A packs have a successor: no tests
#pragma unroll
    for (int i = 0; i < A; ++i) pack(acc[i], true);
  }
#pragma unroll
  for (int i = 0; i < A; ++i)
    if (j + i < cnt) pack(acc[i], j + i + 1 < cnt);
  __syncwarp();
  if constexpr (T::G == 4) {
    const bool hi1 = g & 1, hi2 = g >> 1;
    float q[2 * E];
#pragma unroll
    for (int t = 0; t < 2 * E; ++t)
      q[t] = (hi1 ? acc[0][2 * E + t] : acc[0][t]) +
             __shfl_xor_sync(0xffffffffu, hi1 ? acc[0][t] : acc[0][2 * E + t], T::L);
#pragma unroll
    for (int t = 0; t < E; ++t)
      out[t] = (hi2 ? q[E + t] : q[t]) +
               __shfl_xor_sync(0xffffffffu, hi2 ? q[t] : q[E + t], 2 * T::L);
  } else {
    static_assert(T::G == 2 || T::G == 4, "two or four groups");
    const bool hi = g != 0;
    float q[2][E];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int t = 0; t < E; ++t)
        q[i][t] = (hi ? acc[i % A][E + t] : acc[i % A][t]) +
                  __shfl_xor_sync(0xffffffffu, hi ? acc[i % A][t] : acc[i % A][E + t], T::L);
#pragma unroll
    for (int t = 0; t < E; ++t) out[t] = q[0][t] + q[1][t];
  }
}

// Rows are dealt to teams in the order M.order.  The grid is described by its
// virtual blocks of P_WARPS teams: virtual block vb's team w takes the rows at
// order positions vb * P_WARPS + w + i * (all teams).  A block runs RW virtual
// blocks, so which rows a team takes (and with it the grouping of the
// objective's sums) does not depend on the team's width.
template <int W>
struct RowDeal {
  int vb, w;      // this lane's virtual block and its team in it
  int first, step, rounds;
  __device__ __forceinline__ RowDeal(int rows, int nvb) {
    constexpr int RW = Team<W>::RW;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int u = warp * RW + lane / Team<W>::LANES;
    vb = blockIdx.x * RW + u / P_WARPS;
    w = u % P_WARPS;
    step = nvb * P_WARPS;
    first = vb < nvb ? vb * P_WARPS + w : rows;
    rounds = (rows + step - 1) / step;  // uniform over the grid
  }
  // row of round i, or -1
  __device__ __forceinline__ int row(const DevCSR& M, int i) const {
    const int q = first + i * step;
    if (q >= M.rows || first >= M.rows) return -1;
    return M.order ? __ldg(M.order + q) : q;
  }
};

__device__ double bgn_t(int k, double a, double b, double omega) {
  return a * pow((double)k, omega) + b;
}
// theta_{k+1} (and Nesterov's t_{k+1}) of a slot at index k.
__device__ void next_momentum(SlotState& s) {
  double th = 0.0, t = s.t_cur;
  if (s.momentum == APPGA_MOMENTUM_GN) {
    th = (bgn_t(s.k, s.a, s.b, s.omega) - 1.0) / bgn_t(s.k + 1, s.a, s.b, s.omega);
  } else if (s.momentum == APPGA_MOMENTUM_NESTEROV) {
    const double tn = 0.5 * (1.0 + sqrt(1.0 + 4.0 * t * t));
    th = (t - 1.0) / tn;
    t = tn;
  }
  s.theta_next = th;
  s.t_next = t;
}
__device__ void bset_theta(SlotState& s, double theta) {
  s.theta = theta;
  const float h = (float)theta;
  s.theta_hi = h;
  s.theta_lo = (float)(theta - (double)h);
}

// -------------------------------------------------------------- k_bforward

// One row of per-slot sums per virtual block (its teams in order), in the
// columns of the live slots.
template <int W, class Live>
__device__ __forceinline__ void store_row_sums(const BFwdArgs& a, const float (&dh)[Team<W>::E],
                                               const float (&dl)[Team<W>::E], float (*sum_hi)[W],
                                               float (*sum_lo)[W], const Live& live) {
  using T = Team<W>;
  const int tid = threadIdx.x, lane = tid & 31, sl0 = owned_slot<W>(lane);
  const int team = (tid >> 5) * T::RW + lane / T::LANES;
#pragma unroll
  for (int t = 0; t < T::E; ++t) {
    sum_hi[team][sl0 + t] = dh[t];
    sum_lo[team][sl0 + t] = dl[t];
  }
  __syncthreads();
  for (int q = tid; q < T::RW * W; q += P_THREADS) {
    const int s = q % W, vb = blockIdx.x * T::RW + q / W;
    if (vb >= a.n_spmv_blocks || !live(a.slots[s])) continue;
    float h = 0.f, l = 0.f;
    for (int w = 0; w < P_WARPS; ++w)
      acc_add(h, l, sum_hi[q / W * P_WARPS + w][s], sum_lo[q / W * P_WARPS + w][s]);
    a.fpartial[(size_t)vb * a.Kp + s] = make_float2(h, l);
  }
}

// W: slots the launch works on (every live slot is below it); a.Kp: the row
// stride of the slot-minor arrays, at least W.
template <int W, bool BF16, int NZ>
__global__ void __launch_bounds__(P_THREADS, 2) k_bforward(BFwdArgs a) {
  using T = Team<W>;
  constexpr int E = T::E;
  __shared__ float dsum_hi[P_WARPS * T::RW][W], dsum_lo[P_WARPS * T::RW][W];
  BatchState* bs = a.bst;
  if (a.mode == 0 && bs->remaining == 0) return;  // uniform over the grid
  const int tid = threadIdx.x, lane = tid & 31;
  const int Kp = a.Kp;
  const int G = bs->gstep;
  const float* f = a.f[G % 3];
  float* y_out = a.y[G & 1];
  const float* y_prev = a.y[(G + 1) & 1];
  const bool want = a.track != 0;
  // a first forward phase (of a run, or of admitted slots): f^{k-1} = f^k, so
  // the extrapolated projection is y itself
  const bool first = a.mode != 0;
  auto live = [&](const SlotState& sl) {
    return a.mode == 2 ? sl.fresh : (sl.active && !sl.done);
  };
  const int sl0 = owned_slot<W>(lane), gl0 = gathered_slot<W>(lane);
  int on[E];
  float th_h[E];
  bool any_on = false, gather_on = false;
#pragma unroll
  for (int t = 0; t < E; ++t) {
    const SlotState& sl = a.slots[sl0 + t];
    on[t] = live(sl);
    th_h[t] = first ? 0.f : sl.theta_hi;
    any_on = any_on || on[t];
  }
#pragma unroll
  for (int t = 0; t < T::Q; ++t)
    gather_on = gather_on || live(a.slots[gl0 + t % 4 + t / 4 * T::GSTRIDE]);
  float dh[E], dl[E];
  int hits[E];
#pragma unroll
  for (int t = 0; t < E; ++t) {
    dh[t] = 0.f;
    dl[t] = 0.f;
    hits[t] = 0;
  }
  // the momentum of the next index, so that the pixel phase's last block only
  // copies it: its FP64 powers take about 5 us, here beside the projections
  // of the block's other warps
  if (blockIdx.x == 0 && tid >= P_THREADS - W) {
    SlotState& sl = a.slots[tid - (P_THREADS - W)];
    if (live(sl)) next_momentum(sl);
  }
  const uint64_t pol = evict_first_policy();
  const RowDeal<W> deal(a.A.rows, a.n_spmv_blocks);
  for (int i = 0; i < deal.rounds; ++i) {
    const int row = deal.row(a.A, i);
    float acc[E];
    team_dot<W, BF16, NZ>(a.A, row, f, Kp, lane, gather_on, pol, acc);
    if (row < 0 || !any_on) continue;
    const size_t o = (size_t)row * Kp + sl0;
    float yp[E], gg[E], gm[E], wo[E];
    if (first) {
#pragma unroll
      for (int t = 0; t < E; ++t) yp[t] = acc[t];
    } else {
      vload<E>(y_prev + o, yp);
    }
    vload<E>(a.g + o, gg);
    vload<E>(a.gamma + o, gm);
#pragma unroll
    for (int t = 0; t < E; ++t) {
      wo[t] = 0.f;
      if (!on[t]) continue;
      // y~ = y + theta (y - y_prev); den = max(y~ + gamma, kappa gamma); w = (den - g)/den
      const float yt = first ? acc[t] : fmaf(th_h[t], acc[t] - yp[t], acc[t]);
      float den = yt + gm[t];
      const float fl = 1e-3f * gm[t];
      if (den < fl) {
        den = fl;
        ++hits[t];
      }
      wo[t] = __fdiv_rn(den - gg[t], den);
      if (want) {
        // data term y - g ln(y + gamma) in double-float
        df yg;
        two_sum(acc[t], gm[t], yg.hi, yg.lo);
        const df term = df_add_f(df_neg(df_mul_f(df_log(yg), gg[t])), acc[t]);
        acc_add(dh[t], dl[t], term.hi, term.lo);
      }
    }
    vstore_on<E>(y_out + o, acc, on);
    vstore_on<E>(a.w + o, wo, on);
  }
#pragma unroll
  for (int t = 0; t < E; ++t)
    if (hits[t]) atomicAdd(&a.slots[sl0 + t].guard_hits, (unsigned long long)hits[t]);
  if (!want) return;
  // an admission pass writes only the fresh slots' columns
  store_row_sums<W>(a, dh, dl, dsum_hi, dsum_lo, live);
}

// -------------------------------------------------------------- k_bstencil

// The six fields of B at a pixel from its 3 x 3 neighbourhood x[dr + 1][dc + 1]
// (the forms of the single-slice stencil).
struct BEdges {
  bool r_lo, r_hi, c_lo, c_hi;
};
__device__ __forceinline__ void bfields(const float (&x)[3][3], const BEdges& e, float (&u)[6]) {
  const float dc = x[1][1] - x[1][0], dr = x[1][1] - x[0][1];
  u[0] = e.c_lo ? dc : 0.f;
  u[1] = e.r_lo ? dr : 0.f;
  u[2] = (e.c_lo ? -dc : 0.f) + (e.c_hi ? x[1][2] - x[1][1] : 0.f);
  u[3] = e.c_lo ? ((e.r_lo ? -dc : 0.f) + (e.r_hi ? x[2][1] - x[2][0] : 0.f)) : 0.f;
  u[4] = (e.r_lo ? -dr : 0.f) + (e.r_hi ? x[2][1] - x[1][1] : 0.f);
  u[5] = e.r_lo ? ((e.c_lo ? -dr : 0.f) + (e.c_hi ? x[1][2] - x[0][2] : 0.f)) : 0.f;
}

// B^T grad phi~(B f~) of the current iterates and the regulariser's share of
// Phi(f^k).  A thread owns one slot of one image column and marches down a run
// of rows: the 3 x 3 neighbourhoods of f~ and f^k and the gradient fields of
// its own column stay in registers, and a row's values for the neighbouring
// columns pass through shared memory, slots fastest (no bank conflicts), with
// one barrier per row (the fields of row s - 2 go out with f~ of row s).
// Reading every operand of a point from shared memory instead took 15 passes
// of the L1 pipe per point and slot warp: 255 us at 64 slots of 256 x 256.
// blockIdx.y is the chunk of eight slots; blocks of one x own the same tiles,
// so a slot's sum is grouped the same way whatever its index, and leave their
// row of sums after the projector's.  Runs beside k_bforward (both read only
// the iterates).
__global__ void __launch_bounds__(B_THREADS, 4) k_bstencil(BFwdArgs a) {
  // double-buffered rows: f^k, f~ - f^k and the fields 0, 2, 3, 5
  __shared__ float sK[2][BST_C + 2][BST_S], sD[2][BST_C + 2][BST_S];
  __shared__ float sV[2][4][BST_C + 2][BST_S];
  __shared__ float red_hi[B_THREADS / 32][BST_S], red_lo[B_THREADS / 32][BST_S];
  BatchState* bs = a.bst;
  if (a.mode == 0 && bs->remaining == 0) return;  // uniform over the grid
  const int tid = threadIdx.x, q = tid % BST_S, col = tid / BST_S;
  const int slot = blockIdx.y * BST_S + q, Kp = a.Kp, n = a.n, G = bs->gstep;
  const SlotState& sl = a.slots[slot];
  const bool part = a.mode == 3 ? sl.active
                                : a.mode == 2 ? sl.fresh : (sl.active && !sl.done);
  if (!__syncthreads_or(part)) return;  // no live slot in the chunk
  const bool want = a.track != 0;
  const float* fk = a.f[G % 3] + slot;
  const float *delta = a.delta + slot, *low = a.low + slot;
  float* gR = a.gR + slot;
  const float th = sl.theta_hi;
  const float lam1 = sl.lambda1, lam2 = sl.lambda2, eps = sl.eps, eps2 = eps * eps;
  const int ntx = (n + BST_OUT - 1) / BST_OUT, nty = (n + BST_R - 1) / BST_R;
  float reg_h = 0.f, reg_l = 0.f;
  for (int tile = blockIdx.x; tile < ntx * nty; tile += gridDim.x) {
    const int r0 = (tile / ntx) * BST_R, r1 = min(n, r0 + BST_R);
    const int c = (tile % ntx) * BST_OUT - 2 + col;
    const bool c_in = c >= 0 && c < n;
    const bool out_col = part && c_in && col >= 2 && col < BST_C - 2;
    // f^k and f~ - f^k = theta (f^k - f^{k-1}) + low at rows s - 2 .. s, columns
    // c - 1 .. c + 1
    float k[3][3] = {}, d[3][3] = {};
    // fields of the own column (and the neighbours' where the adjoint reads
    // them): v of row s - 1, w of row s - 2, x of row s - 3
    float v[6] = {}, w0 = 0.f, w0r = 0.f, w1 = 0.f, w2 = 0.f, w2l = 0.f, w2r = 0.f, w3 = 0.f,
          w3r = 0.f, w4 = 0.f, w5 = 0.f, w5l = 0.f;
    float x3 = 0.f, x3r = 0.f, x4 = 0.f, x0 = 0.f, x0r = 0.f, x1 = 0.f, x2 = 0.f, x2l = 0.f,
          x2r = 0.f, x5 = 0.f, x5l = 0.f, y3 = 0.f, y3r = 0.f, y4 = 0.f;
    float nk = 0.f, nd = 0.f, nl = 0.f;  // the next row, in flight
    auto fetch = [&](int r) {
      nk = nd = nl = 0.f;
      if (c_in && r >= 0 && r < n) {
        const size_t o = (size_t)(r * n + c) * Kp;
        nk = fk[o];
        nd = delta[o];
        nl = low[o];
      }
    };
    fetch(r0 - 2);
    for (int s = r0 - 2; s <= r1 + 2; ++s) {
      const int b = s & 1;
      const float vk = nk, vd = fmaf(th, nd, nl);
      sK[b][col + 1][q] = vk;
      sD[b][col + 1][q] = vd;
      // the fields of row s - 2, computed in the last step
      sV[b][0][col + 1][q] = v[0];
      sV[b][1][col + 1][q] = v[2];
      sV[b][2][col + 1][q] = v[3];
      sV[b][3][col + 1][q] = v[5];
      if (s < r1 + 2) fetch(s + 1);
      __syncthreads();
      // rows move up: y is row s - 4, x row s - 3, w row s - 2
      y3 = x3; y3r = x3r; y4 = x4;
      x0 = w0; x0r = w0r; x1 = w1; x2 = w2; x2l = w2l; x2r = w2r;
      x3 = w3; x3r = w3r; x4 = w4; x5 = w5; x5l = w5l;
      w0 = v[0]; w1 = v[1]; w2 = v[2]; w3 = v[3]; w4 = v[4]; w5 = v[5];
      w0r = sV[b][0][col + 2][q];
      w2l = sV[b][1][col][q];
      w2r = sV[b][1][col + 2][q];
      w3r = sV[b][2][col + 2][q];
      w5l = sV[b][3][col][q];
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        k[0][j] = k[1][j];
        k[1][j] = k[2][j];
        d[0][j] = d[1][j];
        d[1][j] = d[2][j];
      }
      k[2][0] = sK[b][col][q];
      k[2][1] = vk;
      k[2][2] = sK[b][col + 2][q];
      d[2][0] = sD[b][col][q];
      d[2][1] = vd;
      d[2][2] = sD[b][col + 2][q];
      // grad phi~ at row i = s - 1
      const int i = s - 1;
      const BEdges e = {i >= 1, i <= n - 2, c >= 1, c <= n - 2};
#pragma unroll
      for (int f = 0; f < 6; ++f) v[f] = 0.f;
      if (c_in && i >= 0 && i < n) {
        // B f~ = B f^k + B (f~ - f^k): f~ itself is never rounded to FP32, and
        // B f^k also serves the regulariser
        float u[6];
        bfields(k, e, u);
        bfields(d, e, v);
#pragma unroll
        for (int f = 0; f < 6; ++f) v[f] += u[f];
        const float n1 = v[0] * v[0] + v[1] * v[1];
        const float n2 = v[2] * v[2] + v[3] * v[3] + v[4] * v[4] + v[5] * v[5];
        const float s1 = lam1 * inv_norm(n1, eps, eps2), s2 = lam2 * inv_norm(n2, eps, eps2);
        v[0] *= s1;
        v[1] *= s1;
#pragma unroll
        for (int f = 2; f < 6; ++f) v[f] *= s2;
        if (want && out_col && i >= r0 && i < r1) {
          const float m1 = u[0] * u[0] + u[1] * u[1];
          const float m2 = u[2] * u[2] + u[3] * u[3] + u[4] * u[4] + u[5] * u[5];
          acc_add(reg_h, reg_l, lam1 * s_eps_f(m1, eps) + lam2 * s_eps_f(m2, eps), 0.f);
        }
      }
      // the adjoint at row o = s - 3: rows o - 1 (y), o (x), o + 1 (w)
      const int o = s - 3;
      if (out_col && o >= r0 && o < r1) {
        const bool r_lo = o >= 1, r_hi = o <= n - 2;
        float sum = 0.f;
        if (e.c_lo) sum += x0;
        if (e.c_hi) sum -= x0r;
        if (r_lo) sum += x1;
        if (r_hi) sum -= w1;
        sum += (e.c_lo ? -(x2 - x2l) : 0.f) + (e.c_hi ? x2r - x2 : 0.f);
        sum += r_lo ? ((e.c_lo ? -(x3 - y3) : 0.f) + (e.c_hi ? x3r - y3r : 0.f)) : 0.f;
        sum += (r_lo ? -(x4 - y4) : 0.f) + (r_hi ? w4 - x4 : 0.f);
        sum += e.c_lo ? ((r_lo ? -(x5 - x5l) : 0.f) + (r_hi ? w5 - w5l : 0.f)) : 0.f;
        gR[(size_t)(o * n + c) * Kp] = sum;
      }
    }
    __syncthreads();  // the row buffers are refilled by the next tile
  }
  if (!want) return;
  // the block's sum of each slot: four columns by shuffles, then the warps in order
#pragma unroll
  for (int o = BST_S; o < 32; o <<= 1)
    acc_add(reg_h, reg_l, __shfl_xor_sync(0xffffffffu, reg_h, o),
            __shfl_xor_sync(0xffffffffu, reg_l, o));
  if (tid % 32 < BST_S) {
    red_hi[tid / 32][q] = reg_h;
    red_lo[tid / 32][q] = reg_l;
  }
  __syncthreads();
  if (tid < BST_S && part) {
    float h = 0.f, l = 0.f;
    for (int w = 0; w < B_THREADS / 32; ++w) acc_add(h, l, red_hi[w][q], red_lo[w][q]);
    a.fpartial[(size_t)(a.n_spmv_blocks + blockIdx.x) * Kp + slot] = make_float2(h, l);
  }
}

// ------------------------------------------------------------- k_bobjective

// Data terms sum y - g ln(y + gamma) of the results of every active slot, with
// y = A f accumulated in double-float as the single-slice objective does (one
// pass over A for all slots: 64 slots of 256 x 256 took 64 projections of 46
// us one by one).  The rows of sums lie as the forward phase's.
template <int W, bool BF16>
__global__ void __launch_bounds__(P_THREADS, 2) k_bobjective(BFwdArgs a) {
  using T = Team<W>;
  constexpr int E = T::E, Q = T::Q, F = Q / 4;
  __shared__ float dsum_hi[P_WARPS * T::RW][W], dsum_lo[P_WARPS * T::RW][W];
  const int lane = threadIdx.x & 31, g = lane % T::LANES / T::L;
  const int sl0 = owned_slot<W>(lane), Kp = a.Kp;
  const float* xl = a.f[a.bst->gstep % 3] + gathered_slot<W>(lane);
  const uint64_t pol = evict_first_policy();
  const RowDeal<W> deal(a.A.rows, a.n_spmv_blocks);
  float dh[E], dl[E];
#pragma unroll
  for (int t = 0; t < E; ++t) dh[t] = dl[t] = 0.f;
  for (int i = 0; i < deal.rounds; ++i) {
    const int row = deal.row(a.A, i);
    float hi[Q], lo[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) hi[q] = lo[q] = 0.f;
    if (row >= 0) {
      const int e = __ldg(a.A.row_ptr + row + 1);
      for (int p = __ldg(a.A.row_ptr + row) + 4 * g; p < e; p += 4 * T::G) {
        const int4 c = ld_stream_i4(a.A.col + p, pol);
        const float4 v = ld_vals<BF16>(a.A, p, pol);
        const int cc[4] = {c.x, c.y, c.z, c.w};
        const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int k = 0; k < F; ++k) {
            const float4 x = *(reinterpret_cast<const float4*>(xl + (unsigned)(cc[u] * Kp)) +
                               k * (T::GSTRIDE / 4));
            acc_fma(hi[4 * k], lo[4 * k], vv[u], x.x);
            acc_fma(hi[4 * k + 1], lo[4 * k + 1], vv[u], x.y);
            acc_fma(hi[4 * k + 2], lo[4 * k + 2], vv[u], x.z);
            acc_fma(hi[4 * k + 3], lo[4 * k + 3], vv[u], x.w);
          }
      }
    }
    __syncwarp();
    // the groups' sums, halving the slots a lane keeps at each exchange
    constexpr int H1 = Q / 2;
    const bool up1 = g & 1;
    float qh[H1], ql[H1];
#pragma unroll
    for (int t = 0; t < H1; ++t) {
      qh[t] = up1 ? hi[H1 + t] : hi[t];
      ql[t] = up1 ? lo[H1 + t] : lo[t];
      acc_add(qh[t], ql[t], __shfl_xor_sync(0xffffffffu, up1 ? hi[t] : hi[H1 + t], T::L),
              __shfl_xor_sync(0xffffffffu, up1 ? lo[t] : lo[H1 + t], T::L));
    }
    if constexpr (T::G == 4) {
      const bool up2 = g >> 1;
#pragma unroll
      for (int t = 0; t < E; ++t) {
        const float sh = __shfl_xor_sync(0xffffffffu, up2 ? qh[t] : qh[E + t], 2 * T::L);
        const float sl = __shfl_xor_sync(0xffffffffu, up2 ? ql[t] : ql[E + t], 2 * T::L);
        qh[t] = up2 ? qh[E + t] : qh[t];
        ql[t] = up2 ? ql[E + t] : ql[t];
        acc_add(qh[t], ql[t], sh, sl);
      }
    }
    if (row < 0) continue;
    float gg[E], gm[E];
    vload<E>(a.g + (size_t)row * Kp + sl0, gg);
    vload<E>(a.gamma + (size_t)row * Kp + sl0, gm);
#pragma unroll
    for (int t = 0; t < E; ++t) {
      const df y = quick_renorm(qh[t], ql[t]);
      const df term = df_add(y, df_neg(df_mul_f(df_log(df_add_f(y, gm[t])), gg[t])));
      acc_add(dh[t], dl[t], term.hi, term.lo);
    }
  }
  store_row_sums<W>(a, dh, dl, dsum_hi, dsum_lo, [](const SlotState& sl) { return sl.active; });
}

// out[2 s] = sum over the first n0 rows, out[2 s + 1] over the next n1 rows, of
// column s (double-float pairs, row stride Kp), in FP64; one block per column.
__global__ void __launch_bounds__(256) k_sum_columns(const float2* __restrict__ rows, int n0,
                                                     int n1, int Kp, double* __restrict__ out) {
  const int s = blockIdx.x;
  for (int part = 0; part < 2; ++part) {
    const int r0 = part ? n0 : 0, r1 = part ? n0 + n1 : n0;
    float h = 0.f, l = 0.f;
    for (int i = r0 + threadIdx.x; i < r1; i += blockDim.x) {
      const float2 v = rows[(size_t)i * Kp + s];
      acc_add(h, l, v.x, v.y);
    }
    const df t = block_sum_acc(h, l);
    if (threadIdx.x == 0) out[2 * s + part] = (double)t.hi + (double)t.lo;
  }
}

// --------------------------------------------------------------- k_bpixel

// Per-slot sums of the forward phase's rows in OBJ_GROUPS groups (rows g,
// g + OBJ_GROUPS, ...), summed by the pixel phase's first blocks; the last
// block adds the group sums.  Every sum runs in four parts combined in order,
// whatever the grid and the slots' number.
constexpr int OBJ_GROUPS = 64;
constexpr int OBJ_PARTS = P_THREADS / MAXK;
__device__ void sum_rows(const float2* rows, int first, int step, int count, int Kp,
                         float (&r_hi)[P_THREADS], float (&r_lo)[P_THREADS]) {
  const int s = threadIdx.x % MAXK, part = threadIdx.x / MAXK;
  float h = 0.f, l = 0.f;
  if (s < Kp) {
#pragma unroll 4
    for (int i = first + part * step; i < count; i += OBJ_PARTS * step) {
      const float2 v = __ldcg(rows + (size_t)i * Kp + s);
      acc_add(h, l, v.x, v.y);
    }
  }
  __syncthreads();
  r_hi[threadIdx.x] = h;
  r_lo[threadIdx.x] = l;
  __syncthreads();
  if (threadIdx.x < MAXK) {
    h = 0.f;
    l = 0.f;
    for (int q = 0; q < OBJ_PARTS; ++q) acc_add(h, l, r_hi[q * MAXK + s], r_lo[q * MAXK + s]);
    r_hi[s] = h;
    r_lo[s] = l;
  }
  __syncthreads();
}

template <int W, bool BF16, int NZ>
__global__ void __launch_bounds__(P_THREADS, 2) k_bpixel(BPixArgs a) {
  using T = Team<W>;
  constexpr int E = T::E;
  __shared__ float r_hi[P_THREADS], r_lo[P_THREADS];
  __shared__ int s_last;
  BatchState* bs = a.bst;
  if (bs->remaining == 0) return;  // uniform over the grid
  const int tid = threadIdx.x, lane = tid & 31;
  const int Kp = a.Kp;
  const int G = bs->gstep;
  const float* fk = a.f[G % 3];
  const float* fkm = a.f[(G + 2) % 3];
  float* fn = a.f[(G + 1) % 3];
  bool any_back = false;
  // every slot's Phi(f^k): the forward phase's rows, first because these
  // blocks start first
  if (a.track)
    for (int g = blockIdx.x; g < OBJ_GROUPS; g += gridDim.x) {
      sum_rows(a.fpartial, g, OBJ_GROUPS, a.n_fpartial, Kp, r_hi, r_lo);
      if (tid < Kp) a.partial[(size_t)g * Kp + tid] = make_float2(r_hi[tid], r_lo[tid]);
    }
  // this lane's slot parameters
  const int sl0 = owned_slot<W>(lane), gl0 = gathered_slot<W>(lane);
  float th[E], beta[E];
  int live[E], kk[E], frz[E], back[E];
  bool gather_live = false;
#pragma unroll
  for (int t = 0; t < E; ++t) {
    const SlotState& sl = a.slots[sl0 + t];
    th[t] = sl.theta_hi;
    beta[t] = sl.beta;
    live[t] = sl.active && !sl.done;
    kk[t] = sl.k;
    frz[t] = sl.freeze_iter;
    back[t] = sl.rollback;
    any_back = any_back || back[t];
  }
#pragma unroll
  for (int t = 0; t < T::Q; ++t) {
    const SlotState& sl = a.slots[gl0 + t % 4 + t / 4 * T::GSTRIDE];
    gather_live = gather_live || (sl.active && !sl.done);
  }
  const uint64_t pol = evict_first_policy();
  int bad = 0;
  const RowDeal<W> deal(a.At.rows, a.n_blocks);
  for (int i = 0; i < deal.rounds; ++i) {
    const int j = deal.row(a.At, i);
    float bp[E];
    team_dot<W, BF16, NZ>(a.At, j, a.w, Kp, lane, gather_live, pol, bp);
    if (j < 0) continue;
    const size_t o = (size_t)j * Kp + sl0;
    float vk[E], vd[E], lo[E], gr[E], out[E];
    vload<E>(fk + o, vk);
    vload<E>(a.delta + o, vd);
    vload<E>(a.low + o, lo);
    vload<E>(a.gR + o, gr);
    const float il = __ldg(a.inv_lambda + j);
#pragma unroll
    for (int t = 0; t < E; ++t) {
      if (!live[t]) {
        // finished or empty slot: carry the image (the previous entry when
        // the slot stopped one step back)
        out[t] = vk[t];
        continue;
      }
      float pk = vk[t];
      if (frz[t] >= 0) {
        if (kk[t] == frz[t]) {
          a.pfreeze[o + t] = vk[t];
        } else if (kk[t] > frz[t]) {
          pk = a.pfreeze[o + t];
        }
      }
      // f^{k+1} = max(f^k + step, 0), step = theta (f^k - f^{k-1}) - p (grad F +
      // grad R): what rounding f^{k+1} to FP32 leaves over is kept in low, and
      // the step itself is the next f^k - f^{k-1}
      const float p = beta[t] * pk * il;
      const float step = __fmaf_rn(th[t], vd[t], -__fmul_rn(p, bp[t] + gr[t]));
      const float full = __fadd_rn(vk[t], lo[t]);
      float xv, rest;
      two_sum(vk[t], __fadd_rn(lo[t], step), xv, rest);
      if (!isfinite(xv)) bad = 1;
      const bool pos = xv > 0.f;
      out[t] = pos ? xv : 0.f;
      vd[t] = pos ? step : -full;
      lo[t] = pos ? rest : 0.f;
    }
    if (any_back) {
#pragma unroll
      for (int t = 0; t < E; ++t)
        if (back[t]) out[t] = fkm[o + t];
    }
    vstore_on<E>(a.delta + o, vd, live);
    vstore_on<E>(a.low + o, lo, live);
    int on[E];
#pragma unroll
    for (int t = 0; t < E; ++t) on[t] = 1;
    vstore_on<E>(fn + o, out, on);
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(&bs->flags, APPGA_FLAG_NONFINITE);
  // Finalise the step in the last block: Phi and the stopping test of every
  // live slot, then its next index and momentum; the global step advances.
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(&bs->ticket_p, 1u) == gridDim.x - 1;
  __syncthreads();
  if (s_last) {
    __threadfence();
    const float *t_hi = r_hi, *t_lo = r_lo;  // the slots' totals
    if (a.track) sum_rows(a.partial, 0, 1, OBJ_GROUPS, Kp, r_hi, r_lo);
    if (tid == 0) bs->ticket_p = 0;
    __shared__ int s_jstop;
    if (a.joint) {
      // volume: the slices are one problem; its objective is the sum of the
      // slots' shares, summed in FP64 in slot order, and one test stops all
      if (tid == 0) {
        double tot = 0.0;
        int kk = -1, k0 = 0;
        double tol = 0.0;
        for (int s = 0; s < Kp; ++s) {
          const SlotState& sl = a.slots[s];
          if (!sl.active || sl.done) continue;
          tot += (double)t_hi[s] + (double)t_lo[s];
          kk = sl.k;
          k0 = sl.k0;
          tol = sl.rel_tol;
        }
        int stop = 0;
        if (kk >= 0 && a.track && bs->phi_tot_k != kk) {
          const double prev = bs->phi_tot_cur;
          const bool consecutive = bs->phi_tot_k == kk - 1;
          bs->phi_tot_prev = prev;
          bs->phi_tot_cur = tot;
          bs->phi_tot_k = kk;
          stop = tol > 0.0 && kk > k0 && consecutive && fabs(tot - prev) <= tol * fabs(prev);
        }
        s_jstop = stop;
      }
      __syncthreads();
    }
    int rem = 0;
    for (int s = tid; s < Kp; s += blockDim.x) {
      SlotState& sl = a.slots[s];
      sl.fresh = 0;
      if (!sl.active || sl.done) {
        sl.rollback = 0;  // its carry above used the previous entry
        continue;
      }
      if (a.track && sl.phi_k != sl.k) {
        const double phi = (double)t_hi[s] + (double)t_lo[s];
        const double prev = sl.phi_cur;
        const bool consecutive = sl.phi_k == sl.k - 1;
        sl.phi_prev = prev;
        sl.phi_cur = phi;
        sl.phi_k = sl.k;
        if (!a.joint && sl.rel_tol > 0.0 && sl.k > sl.k0 && consecutive &&
            fabs(phi - prev) <= sl.rel_tol * fabs(prev)) {
          // f^k is the result; the f^{k+1} written above is not used
          sl.done = 1;
          sl.result_k = sl.k;
          sl.stopped_early = 1;
          sl.rollback = 1;
          continue;
        }
      }
      if (a.joint && s_jstop) {
        // the volume's test fired: f^k of every slice is the result
        sl.done = 1;
        sl.result_k = sl.k;
        sl.stopped_early = 1;
        sl.rollback = 1;
        continue;
      }
      if (sl.k >= sl.k_last) {
        sl.done = 1;
        sl.result_k = sl.k + 1;
      } else {
        ++rem;
      }
      const int k = sl.k;
      sl.k = k + 1;
      sl.t_cur = sl.t_next;
      bset_theta(sl, sl.theta_next);
    }
    static_assert(P_THREADS >= MAXK, "one slot per thread");
    const int tot = __syncthreads_count(rem);
    if (tid == 0) {
      bs->gstep = G + 1;
      bs->remaining = tot;
    }
  }
}

// ----------------------------------------------------------- setup kernels

// Slots marked rollback: copy the previous ring entry into the current one
// (the ring entries of the current global step, read on the device).
__global__ void k_resolve_rollback(const SlotState* slots, const BatchState* bs, float* f0,
                                   float* f1, float* f2, int len, int Kp) {
  const int s = blockIdx.y;
  if (!slots[s].rollback) return;  // uniform over the block
  float* ring[3] = {f0, f1, f2};
  const int G = bs->gstep;
  const float* prev = ring[(G + 2) % 3];
  float* cur = ring[G % 3];
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < len; i += gridDim.x * blockDim.x)
    cur[(size_t)i * Kp + s] = prev[(size_t)i * Kp + s];
}
__global__ void k_clear_rollback(SlotState* slots, int Kp) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < Kp) slots[s].rollback = 0;
}

// theta_{k0} of every slot, or of the fresh slots only (same device
// arithmetic as the step kernel).
__global__ void k_binit_momentum(SlotState* slots, int Kp, int only_fresh) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= Kp) return;
  SlotState& sl = slots[s];
  if (only_fresh && !sl.fresh) return;
  double theta = 0.0, t = 1.0;
  if (sl.momentum == APPGA_MOMENTUM_GN) {
    theta = (bgn_t(sl.k - 1, sl.a, sl.b, sl.omega) - 1.0) / bgn_t(sl.k, sl.a, sl.b, sl.omega);
  } else if (sl.momentum == APPGA_MOMENTUM_NESTEROV) {
    for (int k = 1; k <= sl.k; ++k) {
      const double tn = 0.5 * (1.0 + sqrt(1.0 + 4.0 * t * t));
      theta = (t - 1.0) / tn;
      t = tn;
    }
  }
  bset_theta(sl, theta);
  sl.t_cur = t;
}

// Slot of the k-th slice: ids[k] when a slot list is given, else s0 + k.
__device__ __forceinline__ int slot_of(const int* ids, int s0, int k) {
  return ids ? __ldg(ids + k) : s0 + k;
}

// [K][len] slice-major -> [len][Kp] slot-minor: out[i*Kp + slot(s)] = in[s*len + i].
// Without a slot list the padding slots K .. Kp - 1 get `fill`.  With flag set
// the values are checked on the way: finite and at least 0, or (positive)
// above 0, else *flag becomes 1.
__global__ void k_to_slot_minor(const float* __restrict__ in, int K, int len, float* __restrict__ out,
                                int Kp, int s0, const int* __restrict__ ids, float fill,
                                int positive, int* flag) {
  __shared__ float tile[32][33];
  const int i0 = blockIdx.x * 32, k0 = blockIdx.y * 32;
  int bad = 0;
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int k = k0 + r, i = i0 + threadIdx.x;
    const bool in_range = k < K && i < len;
    const float v = in_range ? in[(size_t)k * len + i] : fill;
    if (in_range && !(isfinite(v) && (positive ? v > 0.f : v >= 0.f))) bad = 1;
    tile[r][threadIdx.x] = v;
  }
  if (__syncthreads_or(bad) && flag != nullptr && threadIdx.x == 0 && threadIdx.y == 0)
    atomicOr(flag, 1);
  const int top = ids ? K : Kp - s0;
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int i = i0 + r, k = k0 + threadIdx.x;
    if (i < len && k < top) out[(size_t)i * Kp + slot_of(ids, s0, k)] = tile[threadIdx.x][r];
  }
}
// out[s*len + i] = in[i*Kp + slot(s)] for s < K, in the ring entry of the
// current global step.
__global__ void k_from_slot_minor(const float* f0, const float* f1, const float* f2,
                                  const BatchState* bst, int K, int len, int Kp, int s0,
                                  const int* __restrict__ ids, float* __restrict__ out) {
  __shared__ float tile[32][33];
  const float* ring[3] = {f0, f1, f2};
  const float* in = ring[bst->gstep % 3];
  const int i0 = blockIdx.x * 32, k0 = blockIdx.y * 32;
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int i = i0 + r, k = k0 + threadIdx.x;
    tile[r][threadIdx.x] = (i < len && k < K) ? in[(size_t)i * Kp + slot_of(ids, s0, k)] : 0.f;
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int k = k0 + r, i = i0 + threadIdx.x;
    if (k < K && i < len) out[(size_t)k * len + i] = tile[threadIdx.x][r];
  }
}
// Sets column s of a [len][Kp] array to v for s in [s0, s1).
__global__ void k_fill_slots(float* out, int len, int Kp, int s0, int s1, float v) {
  const int w = s1 - s0;
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < (size_t)len * w;
       t += (size_t)gridDim.x * blockDim.x)
    out[(t / w) * Kp + s0 + t % w] = v;
}

// Per-slot initial image TMC_s * 1_disk (Sec. 4.1) for the slots of K slices
// (s0 + k, or ids[k]) from slice-major g, gamma ([K][m]): ACT_PARTS blocks per
// slice sum g - gamma, then the images are filled a row of slots at a time (one
// block per slice did both: 192 us for 64 slices of 256 x 256, 12 us now).
constexpr int ACT_PARTS = 16;
__global__ void __launch_bounds__(256) k_bactc(const float* __restrict__ g,
                                               const float* __restrict__ gamma, int m,
                                               float2* __restrict__ parts) {
  const int k = blockIdx.y;
  float h = 0.f, l = 0.f;
#pragma unroll 4
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
    acc_add(h, l, g[(size_t)k * m + i], 0.f);
    acc_add(h, l, -gamma[(size_t)k * m + i], 0.f);
  }
  const df t = block_sum_acc(h, l);
  if (threadIdx.x == 0) parts[k * ACT_PARTS + blockIdx.x] = make_float2(t.hi, t.lo);
}
// f_cur and, if not NULL, f_prev; delta and low become 0; without a slot list
// the padding slots get 0.
__global__ void __launch_bounds__(256) k_binit_image(const float2* __restrict__ parts, int n,
                                                     int n_angles, long long npfov, int K, int Kp,
                                                     int s0, const int* __restrict__ ids,
                                                     float* __restrict__ f_cur,
                                                     float* __restrict__ f_prev,
                                                     float* __restrict__ delta,
                                                     float* __restrict__ low) {
  __shared__ float s_tmc[MAXK];
  for (int k = threadIdx.x; k < K; k += blockDim.x) {
    float h = 0.f, l = 0.f;
    for (int q = 0; q < ACT_PARTS; ++q) {
      const float2 v = parts[k * ACT_PARTS + q];
      acc_add(h, l, v.x, v.y);
    }
    s_tmc[k] = (float)(((double)h + (double)l) / ((double)npfov * (double)n_angles));
  }
  __syncthreads();
  const int cols = ids ? K : Kp - s0;
  const size_t total = (size_t)n * n * cols;
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total;
       t += (size_t)gridDim.x * blockDim.x) {
    const int j = (int)(t / cols), k = (int)(t % cols);
    const int r = j / n, c = j % n;
    const long long dx = 2ll * c + 1 - n, dy = 2ll * r + 1 - n;
    const float v = k < K && dx * dx + dy * dy <= (long long)n * n ? s_tmc[k] : 0.f;
    const size_t o = (size_t)j * Kp + slot_of(ids, s0, k);
    f_cur[o] = v;
    if (f_prev) f_prev[o] = v;
    delta[o] = 0.f;
    low[o] = 0.f;
  }
}


int sm_count() { return current_sm_count(); }

// Virtual blocks of the forward phase's projector rows.
int fw_blocks(const BFwdArgs& a) {
  const int nb = (a.A.rows + P_WARPS - 1) / P_WARPS;
  return std::min(nb, sm_count() * clamp_per_sm(a.spmv_per_sm, kSpmvPerSm));
}
// Stencil blocks per slot chunk: equal tile counts per block.
int st_blocks(const BFwdArgs& a) {
  if (a.no_stencil) return 0;
  const int tiles = ((a.n + BST_OUT - 1) / BST_OUT) * ((a.n + BST_R - 1) / BST_R);
  const int cap = sm_count() * clamp_per_sm(a.stencil_per_sm, kStencilPerSm);
  const int per = (tiles + cap - 1) / cap;
  return (tiles + per - 1) / per;
}

// Gather probe: the batched projectors' inner loop alone.  Every row of M is
// reduced against the W-wide slot-minor rows of x by team_dot, dealt to the
// teams as in the projections, with no epilogue, stencil or pixel update.
template <int W>
__global__ void __launch_bounds__(P_THREADS, 2) k_gather_probe(DevCSR M, const float* __restrict__ x,
                                                               int nvb, float* __restrict__ sink) {
  const int lane = threadIdx.x & 31;
  const uint64_t pol = evict_first_policy();
  const RowDeal<W> deal(M.rows, nvb);
  float s = 0.f;
  for (int i = 0; i < deal.rounds; ++i) {
    float acc[Team<W>::E];
    team_dot<W, false, 4>(M, deal.row(M, i), x, W, lane, true, pol, acc);
#pragma unroll
    for (int t = 0; t < Team<W>::E; ++t) s += acc[t];
  }
  if (s == 1.0e38f) sink[blockIdx.x] = s;  // keeps the loads; the value is never used
}

template <int W>
int blocks_of(int nvb) {
  return (nvb + Team<W>::RW - 1) / Team<W>::RW;
}

template <int W>
cudaError_t bforward_w(const BFwdArgs& a, cudaStream_t s) {
  const bool g4 = a.gather_rows == 4;
  void (*kern)(BFwdArgs) = a.use_bf16 ? (g4 ? k_bforward<W, true, 2> : k_bforward<W, true, 4>)
                                      : (g4 ? k_bforward<W, false, 2> : k_bforward<W, false, 4>);
  kern<<<blocks_of<W>(a.n_spmv_blocks), P_THREADS, 0, s>>>(a);
  return cudaGetLastError();
}
template <int W>
cudaError_t bpixel_w(const BPixArgs& a, cudaStream_t s) {
  const bool g4 = a.gather_rows == 4;
  void (*kern)(BPixArgs) = a.use_bf16 ? (g4 ? k_bpixel<W, true, 2> : k_bpixel<W, true, 4>)
                                      : (g4 ? k_bpixel<W, false, 2> : k_bpixel<W, false, 4>);
  kern<<<blocks_of<W>(a.n_blocks), P_THREADS, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace

// Largest grid of the batched kernels: at most kMaxPerSm SpMV and kMaxPerSm
// stencil blocks per SM (the launchers clamp the tuned values).
int batch_max_blocks() { return sm_count() * 2 * kMaxPerSm + 64; }

int bforward_grid(const BFwdArgs& a) { return fw_blocks(a) + st_blocks(a); }

cudaError_t launch_resolve_rollback(const BFwdArgs& a, cudaStream_t s) {
  const int len = a.n * a.n;
  dim3 grid((len + 255) / 256 < 64 ? (len + 255) / 256 : 64, a.Kp);
  k_resolve_rollback<<<grid, 256, 0, s>>>(a.slots, a.bst, a.f[0], a.f[1], a.f[2], len, a.Kp);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // cleared by a second launch: every block above has read the mark first
  k_clear_rollback<<<(a.Kp + 127) / 128, 128, 0, s>>>(a.slots, a.Kp);
  return cudaGetLastError();
}

cudaError_t launch_bforward(const BFwdArgs& a0, cudaStream_t s) {
  cudaError_t e = ensure_tables();
  if (e != cudaSuccess) return e;
  BFwdArgs a = a0;
  a.n_spmv_blocks = fw_blocks(a);
  switch (a.width) {
    case 8: return bforward_w<8>(a, s);
    case 16: return bforward_w<16>(a, s);
    case 32: return bforward_w<32>(a, s);
    case 64: return bforward_w<64>(a, s);
    case 128: return bforward_w<128>(a, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_bstencil(const BFwdArgs& a0, cudaStream_t s) {
  BFwdArgs a = a0;
  a.n_spmv_blocks = fw_blocks(a);
  const int nst = st_blocks(a);
  if (nst == 0) return cudaSuccess;
  k_bstencil<<<dim3(nst, a.width / BST_S), B_THREADS, 0, s>>>(a);
  return cudaGetLastError();
}

namespace {
template <int W>
cudaError_t bobjective_w(const BFwdArgs& a, cudaStream_t s) {
  if (a.use_bf16)
    k_bobjective<W, true><<<blocks_of<W>(a.n_spmv_blocks), P_THREADS, 0, s>>>(a);
  else
    k_bobjective<W, false><<<blocks_of<W>(a.n_spmv_blocks), P_THREADS, 0, s>>>(a);
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_bobjective(const BFwdArgs& a0, int K, double* out, cudaStream_t s) {
  cudaError_t e = ensure_tables();
  if (e != cudaSuccess) return e;
  BFwdArgs a = a0;
  a.mode = 3;
  a.track = 1;
  a.n_spmv_blocks = fw_blocks(a);
  switch (a.width) {
    case 8: e = bobjective_w<8>(a, s); break;
    case 16: e = bobjective_w<16>(a, s); break;
    case 32: e = bobjective_w<32>(a, s); break;
    case 64: e = bobjective_w<64>(a, s); break;
    case 128: e = bobjective_w<128>(a, s); break;
    default: e = cudaErrorInvalidValue;
  }
  if (e == cudaSuccess) e = launch_bstencil(a, s);
  if (e != cudaSuccess) return e;
  k_sum_columns<<<K, 256, 0, s>>>(a.fpartial, a.n_spmv_blocks, st_blocks(a), a.Kp, out);
  return cudaGetLastError();
}

cudaError_t launch_gather_probe(const DevCSR& M, const float* x, int Kp, float* sink,
                                int blocks_per_sm, cudaStream_t s) {
  if (blocks_per_sm < 1 || blocks_per_sm > kMaxPerSm) return cudaErrorInvalidValue;
  const int grid = std::min((M.rows + P_WARPS - 1) / P_WARPS, sm_count() * blocks_per_sm);
  switch (Kp) {
    case 32: k_gather_probe<32><<<grid, P_THREADS, 0, s>>>(M, x, grid, sink); break;
    case 64: k_gather_probe<64><<<grid, P_THREADS, 0, s>>>(M, x, grid, sink); break;
    case 128: k_gather_probe<128><<<grid, P_THREADS, 0, s>>>(M, x, grid, sink); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_bpixel(const BPixArgs& a0, cudaStream_t s) {
  BPixArgs a = a0;
  a.n_blocks = std::min((a.At.rows + P_WARPS - 1) / P_WARPS,
                        sm_count() * clamp_per_sm(a.blocks_per_sm, kPixelPerSm));
  switch (a.width) {
    case 8: return bpixel_w<8>(a, s);
    case 16: return bpixel_w<16>(a, s);
    case 32: return bpixel_w<32>(a, s);
    case 64: return bpixel_w<64>(a, s);
    case 128: return bpixel_w<128>(a, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_binit_momentum(SlotState* slots, int Kp, bool only_fresh, cudaStream_t s) {
  k_binit_momentum<<<(Kp + 127) / 128, 128, 0, s>>>(slots, Kp, only_fresh ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_to_slot_minor(const float* in, int K, int len, float* out, int Kp, int s0,
                                 const int* ids, cudaStream_t s, float fill, bool positive,
                                 int* flag) {
  if (K <= 0) return cudaSuccess;
  const int cols = ids ? K : Kp - s0;
  dim3 grid((len + 31) / 32, (cols + 31) / 32), block(32, 8);
  k_to_slot_minor<<<grid, block, 0, s>>>(in, K, len, out, Kp, s0, ids, fill, positive ? 1 : 0,
                                         flag);
  return cudaGetLastError();
}

cudaError_t launch_from_slot_minor(const BFwdArgs& a, int K, int s0, const int* ids, float* out,
                                   cudaStream_t s) {
  if (K <= 0) return cudaSuccess;
  const int len = a.n * a.n;
  dim3 grid((len + 31) / 32, (K + 31) / 32), block(32, 8);
  k_from_slot_minor<<<grid, block, 0, s>>>(a.f[0], a.f[1], a.f[2], a.bst, K, len, a.Kp, s0, ids,
                                           out);
  return cudaGetLastError();
}

cudaError_t launch_fill_slots(float* out, int len, int Kp, int s0, int s1, float v,
                              cudaStream_t s) {
  if (s1 <= s0) return cudaSuccess;
  k_fill_slots<<<256, 256, 0, s>>>(out, len, Kp, s0, s1, v);
  return cudaGetLastError();
}

cudaError_t launch_binit_image(const float* g, const float* gamma, int m, int n, int n_angles,
                               long long npfov, int K, int Kp, int s0, const int* ids,
                               float2* scratch, float* f_cur, float* f_prev, float* delta,
                               float* low, cudaStream_t s) {
  if (K <= 0) return cudaSuccess;
  k_bactc<<<dim3(ACT_PARTS, K), 256, 0, s>>>(g, gamma, m, scratch);
  const long long total = (long long)n * n * (ids ? K : Kp - s0);
  const int grid = (int)std::min<long long>((total + 255) / 256, sm_count() * 8LL);
  k_binit_image<<<grid, 256, 0, s>>>(scratch, n, n_angles, npfov, K, Kp, s0, ids, f_cur, f_prev,
                                      delta, low);
  return cudaGetLastError();
}

}  // namespace appga
