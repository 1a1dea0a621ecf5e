// Batched CUDA kernels: K independent slices (slots) that share one system
// matrix run the APPGA iteration together, so every nonzero of A and A^T is
// read once per iteration for all K right-hand sides (SpMM).
//
// Layout (slot-minor): images f[j][s], sinograms y[i][s], w[i][s], g[i][s],
// rows of Kp slots.  A launch works on as many slots as are held: 8, 16, 32, 64
// or twice 64.  The projections take the matrices in blocks of four neighbouring
// rows (DevQuad), so that a gathered row serves up to four of them from
// registers; QTeam says how a warp shares a block and what bounds it.  Blocks
// follow a Z-order curve (pixels, or rays by angle and bin), so the blocks of an
// SM gather for neighbouring rows and meet in L1.  The per-(row, slot) epilogues
// match the single-slice kernels (Eq. APPGAiter, Eq. EM, Sec. 2.2); the SHOITV
// stencil is a kernel of its own that runs beside the forward projection.
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
#include <type_traits>

#include "appga_internal.h"
#include "batched_internal.h"
#include "device_common.cuh"

namespace appga {
namespace {

constexpr int B_THREADS = 256;               // stencil blocks (and set-up kernels)
constexpr int MAXK = 128;                    // largest padded batch
// Projector blocks: four warps, four blocks per SM (128 registers per thread:
// a step's gathers are in flight at once, which gains more than more warps with
// half of them would; eight-warp blocks are slower, their last warps idle more).
constexpr int Q_THREADS = 128;
constexpr int Q_WARPS = Q_THREADS / 32;
constexpr int Q_PER_SM = 4;
// Blocks of the objective's double-float projections.
constexpr int P_THREADS = 512;
constexpr int P_WARPS = P_THREADS / 32;
constexpr int kMaxPerSm = 16;                // upper bound of the tuned values
__host__ __forceinline__ int clamp_per_sm(int v, int dflt) {
  return v <= 0 ? dflt : (v > kMaxPerSm ? kMaxPerSm : v);
}
// Virtual blocks per SM when no tuned schedule is given: more than are resident
// at once, so the block scheduler levels the tail.
constexpr int kSpmvPerSm = 16;
constexpr int kPixelPerSm = 16;
constexpr int kObjectivePerSm = 8;
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
__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}
// Stores the elements whose bit is set in `on` (one vector store when all are).
template <int V>
__device__ __forceinline__ void vstore(float* p, const float (&x)[V], unsigned on) {
  if (on == (1u << V) - 1) {
    if constexpr (V == 1) {
      *p = x[0];
    } else if constexpr (V == 2) {
      *reinterpret_cast<float2*>(p) = make_float2(x[0], x[1]);
    } else {
      *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
    }
  } else {
#pragma unroll
    for (int t = 0; t < V; ++t)
      if (on >> t & 1) p[t] = x[t];
  }
}
// Two FP32 values in one 64-bit register pair, and a += w x on both (each
// rounded once, as fmaf).
__device__ __forceinline__ unsigned long long pair_of(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void split(unsigned long long v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ void fma2(unsigned long long& a, unsigned long long w,
                                     unsigned long long x) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(a) : "l"(w), "l"(x));
}
// The four rows' values at union column o.
template <bool BF16>
__device__ __forceinline__ float4 ld_quad(const DevQuad& M, size_t o, uint64_t pol) {
  if constexpr (BF16) {
    const uint2 u = ld_stream_u2(M.vals_bf16 + o, pol);
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u),
                       __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
  } else {
    return ld_stream_f4(reinterpret_cast<const float*>(M.vals + o), pol);
  }
}

// The objective's double-float projections take one row at a time from the
// CSR: how the lanes of a warp share a row whose products fill W <= 64 slots (a
// grid of two in y covers 128).  A lane holds Q slots (Q/4 16-byte loads per
// gathered row), L lanes make a group that covers the W slots, and the four
// groups of a row's team take the row's 4-entry packs in turn, RW rows of the
// warp at a time.  The row's sum is that of four partial sums, p_i over the
// packs k = i (mod 4) in order, as (p0 + p1) + (p2 + p3), so the results do not
// depend on W.  Eight slots per lane because the load of a pack's columns or values, which
// a group's lanes make at one address, still takes the L1 pipe four passes
// (a 16-byte load is served in quarter warps): with four groups a warp those
// passes feed 16 entries.
template <int W>
struct Team {
  static constexpr int Q = W >= 16 ? 8 : 4;
  static constexpr int L = W / Q;
  static constexpr int G = 4;
  static constexpr int LANES = L * G;
  static constexpr int RW = 32 / LANES;
  static constexpr int E = Q / G;  // slots a lane owns after the reduction
  static constexpr int GSTRIDE = 4 * L;
  static_assert(LANES <= 32, "a team is part of a warp");
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

// How the kernels' warps share the layout's blocks of four rows (DevQuad): a
// lane holds Q slots, L lanes make a group that covers the W slots, and the S
// groups of a block's team take the block's packs of four union columns in turn
// (pack k: group k mod S), each summing all four rows.  The groups' sums are
// added pairwise along the bits of the group's index, so the results do not
// depend on W.  A narrow team is part of a warp, RW of them, a wide one NWQ
// warps of GW groups.
//
// The L1 pipe bounds these kernels on large matrices (S = 4).  Per union column
// it passes W/32 lines of the gathered row and, because a 16-byte load is
// served in quarter warps even where its lanes share an address, a quarter pass
// for the column and one for the four values (four groups, four passes a load).
// A union column serves 2.0 pixels of the back-projection, or 1.5 rays of the
// forward projection, so at 64 slots an entry costs 1.6 or 2.2 passes against
// 3.0 with one row per warp: 64 slots of 256 x 256 take 167 and 216 us against
// 247 and 257 us.  Small matrices have too few blocks to fill the chip and each
// team's chain of packs is what they wait for: S = 16 quarters it.
constexpr int QROWS = 4;
template <int W, int S>
struct QTeam {
  static constexpr int Q = W >= 64 ? 8 : 4;
  static constexpr int F = Q / 4;  // 16-byte pieces of a gathered row per lane
  static constexpr int U = Q == 4 ? 2 : 1;  // packs a lane gathers per step (NZ = 4)
  static constexpr int L = W / Q;
  static constexpr int STRIDE = 4 * L;  // slots between a lane's pieces
  static constexpr int GW = S < 32 / L ? S : 32 / L;
  static constexpr int NWQ = S / GW;
  static constexpr int LANES = GW * L;
  static constexpr int RW = 32 / LANES;
  static constexpr int TB = Q_WARPS / NWQ * RW;  // teams of a thread block
  static constexpr int TV = S == 4 ? 4 : 1;      // teams of a virtual block
  // after the reduction a lane owns E slots of one row, in pieces of V
  static constexpr int EW = Q / (GW / 4);
  static constexpr int E = EW / NWQ;
  static constexpr int V = E < 4 ? E : 4;
  static_assert(GW >= 4 && E >= 1 && TB % TV == 0, "two exchanges halve the rows");
};
// A lane's place in its team.
template <int W, int S>
struct QLane {
  int lane, warp, team, g, wq, row, slot;  // team of the block; group in the warp; warp in the
                                           // team; owned row and first owned slot
  __device__ __forceinline__ QLane() {
    using T = QTeam<W, S>;
    lane = threadIdx.x & 31;
    warp = threadIdx.x >> 5;
    team = warp / T::NWQ * T::RW + lane / T::LANES;
    g = lane % T::LANES / T::L;
    wq = warp % T::NWQ;
    row = 2 * (g & 1) + (g >> 1 & 1);
    int raw = T::E * wq;
    if (T::GW >= 8) raw += T::Q / 2 * (g >> 2 & 1);
    if (T::GW >= 16) raw += T::Q / 4 * (g >> 3 & 1);
    slot = gathered() + raw / 4 * T::STRIDE + raw % 4;
  }
  // first of the lane's gathered slots (pieces of four, STRIDE apart)
  __device__ __forceinline__ int gathered() const { return 4 * (lane % QTeam<W, S>::L); }
};

// Block b (negative: none) of M times the columns of X ([cols][stride]): the
// lane's group's sums of its gathered slots for the four rows, as pairs of
// neighbouring slots for the two-wide FP32 FMA.  A lane gathers NZ (2 or 4)
// columns per step; `on`: some of its slots is wanted.
template <int W, int S, bool BF16, int NZ>
__device__ __forceinline__ void quad_sums(const DevQuad& M, int b, const float* __restrict__ X,
                                          int stride, const QLane<W, S>& me, bool on, uint64_t pol,
                                          unsigned long long (&acc2)[QROWS][QTeam<W, S>::Q / 2]) {
  using T = QTeam<W, S>;
  constexpr int Q = T::Q, F = T::F;
  int k = 0, e = 0;
  if (b >= 0 && on) {
    k = __ldg(M.off + b) + me.wq * T::GW + me.g;
    e = __ldg(M.off + b + 1);
  }
  const float* xl = X + me.gathered();
#pragma unroll
  for (int r = 0; r < QROWS; ++r)
#pragma unroll
    for (int q = 0; q < Q / 2; ++q) acc2[r][q] = 0ull;
  constexpr int U = NZ == 4 ? T::U : 1;  // (a pack's products stay in its entries' order)
  int4 c[U];
#pragma unroll
  for (int p = 0; p < U; ++p) {
    c[p] = make_int4(0, 0, 0, 0);
    if (k + S * p < e) c[p] = ld_stream_i4(reinterpret_cast<const int32_t*>(M.cols + k + S * p), pol);
  }
  // one step: U packs' gathers, the next U packs' columns, the products
  auto step = [&](auto full) {
    // the stream is two steps ahead in L2 (the loads below would otherwise
    // wait for DRAM: 207 us of back-projection at 64 slots of 256 x 256, 189 so)
    if constexpr (BF16)
      prefetch_l2(M.vals_bf16 + 4 * (size_t)(k + 2 * S * U));
    else
      prefetch_l2(M.vals + 4 * (size_t)(k + 2 * S * U));
    prefetch_l2(M.cols + (k + 2 * S * U));
#pragma unroll
    for (int h = 0; h < 4; h += NZ) {
      ulonglong2 x[U][NZ][F];
      float4 v[U][NZ];
#pragma unroll
      for (int p = 0; p < U; ++p) {
        if (!full.value && k + S * p >= e) continue;
        const int cc[4] = {c[p].x, c[p].y, c[p].z, c[p].w};
#pragma unroll
        for (int u = 0; u < NZ; ++u) {
#pragma unroll
          for (int i = 0; i < F; ++i)
            x[p][u][i] =
                __ldg(reinterpret_cast<const ulonglong2*>(xl + (unsigned)(cc[h + u] * stride)) +
                      i * (T::STRIDE / 4));
          v[p][u] = ld_quad<BF16>(M, 4 * (size_t)(k + S * p) + h + u, pol);
        }
      }
      if (h + NZ == 4) {
#pragma unroll
        for (int p = 0; p < U; ++p)
          if (k + S * (U + p) < e)
            c[p] = ld_stream_i4(reinterpret_cast<const int32_t*>(M.cols + k + S * (U + p)), pol);
      }
#pragma unroll
      for (int p = 0; p < U; ++p) {
        if (!full.value && k + S * p >= e) continue;
#pragma unroll
        for (int u = 0; u < NZ; ++u) {
          const float vv[QROWS] = {v[p][u].x, v[p][u].y, v[p][u].z, v[p][u].w};
#pragma unroll
          for (int r = 0; r < QROWS; ++r) {
            const unsigned long long w = pair_of(vv[r], vv[r]);
#pragma unroll
            for (int i = 0; i < F; ++i) {
              fma2(acc2[r][2 * i], w, x[p][u][i].x);
              fma2(acc2[r][2 * i + 1], w, x[p][u][i].y);
            }
          }
        }
      }
    }
    k += S * U;
  };
  while (k + S * (U - 1) < e) step(std::true_type{});
  if (U > 1 && k < e) step(std::false_type{});
}
// The groups' sums added up: the lane's E owned slots of its row.  All threads of
// the block take part; each exchange halves the rows, then the slots a lane
// keeps.  s_x: shared, 2 x Q_WARPS x EW x 32 floats where teams span warps;
// `parity` alternates between its halves.
template <int W, int S>
__device__ __forceinline__ void quad_reduce(
    const unsigned long long (&acc2)[QROWS][QTeam<W, S>::Q / 2], const QLane<W, S>& me,
    float* s_x, int parity, float (&out)[QTeam<W, S>::E]) {
  using T = QTeam<W, S>;
  constexpr int Q = T::Q, EW = T::EW;
  float acc[QROWS][Q];
#pragma unroll
  for (int r = 0; r < QROWS; ++r)
#pragma unroll
    for (int q = 0; q < Q / 2; ++q) split(acc2[r][q], acc[r][2 * q], acc[r][2 * q + 1]);
  __syncwarp();
  const bool up0 = me.g & 1, up1 = me.g >> 1 & 1, up2 = me.g >> 2 & 1, up3 = me.g >> 3 & 1;
  float q[2][Q], v[Q];
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int t = 0; t < Q; ++t)
      q[r][t] = (up0 ? acc[2 + r][t] : acc[r][t]) +
                __shfl_xor_sync(0xffffffffu, up0 ? acc[r][t] : acc[2 + r][t], T::L);
#pragma unroll
  for (int t = 0; t < Q; ++t)
    v[t] = (up1 ? q[1][t] : q[0][t]) +
           __shfl_xor_sync(0xffffffffu, up1 ? q[0][t] : q[1][t], 2 * T::L);
  if constexpr (T::GW >= 8) {
#pragma unroll
    for (int t = 0; t < Q / 2; ++t)
      v[t] = (up2 ? v[Q / 2 + t] : v[t]) +
             __shfl_xor_sync(0xffffffffu, up2 ? v[t] : v[Q / 2 + t], 4 * T::L);
  }
  if constexpr (T::GW >= 16) {
#pragma unroll
    for (int t = 0; t < Q / 4; ++t)
      v[t] = (up3 ? v[Q / 4 + t] : v[t]) +
             __shfl_xor_sync(0xffffffffu, up3 ? v[t] : v[Q / 4 + t], 8 * T::L);
  }
  if constexpr (T::NWQ == 1) {
#pragma unroll
    for (int t = 0; t < T::E; ++t) out[t] = v[t];
  } else {
    float* buf = s_x + parity * Q_WARPS * EW * 32;
#pragma unroll
    for (int t = 0; t < EW; ++t) buf[(me.warp * EW + t) * 32 + me.lane] = v[t];
    __syncthreads();
    const int w0 = me.warp - me.wq;
#pragma unroll
    for (int t = 0; t < T::E; ++t) {
      float x[T::NWQ];
#pragma unroll
      for (int w = 0; w < T::NWQ; ++w)
        x[w] = buf[((w0 + w) * EW + T::E * me.wq + t) * 32 + me.lane];
      out[t] = T::NWQ == 2 ? x[0] + x[1] : (x[0] + x[1]) + (x[2 % T::NWQ] + x[3 % T::NWQ]);
    }
  }
}
template <int W, int S>
constexpr int kReduceFloats = QTeam<W, S>::NWQ > 1 ? 2 * Q_WARPS * QTeam<W, S>::EW * 32 : 1;

// Blocks of the layout are dealt to teams in order.  The grid is described by
// its virtual blocks of TV teams: virtual block vb's team w takes blocks
// vb TV + w + i (all teams).  A thread block runs TB / TV virtual blocks, so
// which rows a team takes (and with it the grouping of the objective's sums)
// does not depend on the team's width.
template <int W, int S>
struct QuadDeal {
  int vb, first, step, rounds;
  __device__ __forceinline__ QuadDeal(const QLane<W, S>& me, int blocks, int nvb) {
    using T = QTeam<W, S>;
    vb = blockIdx.x * (T::TB / T::TV) + me.team / T::TV;
    step = nvb * T::TV;
    first = vb < nvb ? vb * T::TV + me.team % T::TV : blocks;
    rounds = (blocks + step - 1) / step;  // uniform over the grid
  }
  // starts the loads of the first block's extent and rows
  __device__ __forceinline__ void warm(const DevQuad& M) const {
    if (first < M.blocks) {
      asm volatile("prefetch.global.L1 [%0];" ::"l"(M.off + first));
      asm volatile("prefetch.global.L1 [%0];" ::"l"(M.rows + QROWS * first));
    }
  }
  __device__ __forceinline__ int block(const DevQuad& M, int i) const {
    const int q = first + i * step;
    return first < M.blocks && q < M.blocks ? q : -1;
  }
};

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
  const int s0 = blockIdx.y * W;
  for (int q = tid; q < T::RW * W; q += P_THREADS) {
    const int s = q % W, vb = blockIdx.x * T::RW + q / W;
    if (vb >= a.n_spmv_blocks || !live(a.slots[s0 + s])) continue;
    float h = 0.f, l = 0.f;
    for (int w = 0; w < P_WARPS; ++w)
      acc_add(h, l, sum_hi[q / W * P_WARPS + w][s], sum_lo[q / W * P_WARPS + w][s]);
    a.fpartial[(size_t)vb * a.Kp + s0 + s] = make_float2(h, l);
  }
}

// Slots are worked on W at a time: blockIdx.y takes those from y W on (every
// live slot is below gridDim.y W); a.Kp: the row stride of the slot-minor
// arrays.
template <int W, int S, bool BF16, int NZ>
__global__ void __launch_bounds__(Q_THREADS, Q_PER_SM) k_bforward(BFwdArgs a) {
  using T = QTeam<W, S>;
  constexpr int E = T::E, V = T::V;
  __shared__ float s_th[W];
  __shared__ float d_hi[T::TB * QROWS][W], d_lo[T::TB * QROWS][W];  // data terms by team and row
  __shared__ float s_x[kReduceFloats<W, S>];
  BatchState* bs = a.bst;
  const int remaining = bs->remaining, G = bs->gstep;
  const QLane<W, S> me;
  const QuadDeal<W, S> deal(me, a.QA.blocks, a.n_spmv_blocks);
  deal.warm(a.QA);
  const int tid = threadIdx.x;
  const int Kp = a.Kp, s0 = blockIdx.y * W;
  const float* f = a.f[G % 3] + s0;
  float* y_out = a.y[G & 1];
  const float* y_prev = a.y[(G + 1) & 1];
  const bool want = a.track != 0;
  // a first forward phase (of a run, or of admitted slots): f^{k-1} = f^k, so
  // the extrapolated projection is y itself
  const bool first = a.mode != 0;
  SlotState* slots = a.slots + s0;
  auto live = [&](const SlotState& sl) {
    return a.mode == 2 ? sl.fresh : (sl.active && !sl.done);
  };
  unsigned on = 0;  // the lane's live owned slots
  bool gather_on = false;
#pragma unroll
  for (int t = 0; t < E; ++t)
    on |= live(slots[me.slot + t / V * T::STRIDE + t % V]) ? 1u << t : 0u;
#pragma unroll
  for (int t = 0; t < T::Q; ++t)
    gather_on = gather_on || live(slots[me.gathered() + t / 4 * T::STRIDE + t % 4]);
  for (int t = tid; t < W; t += Q_THREADS) s_th[t] = first ? 0.f : slots[t].theta_hi;
  if (a.mode == 0 && remaining == 0) return;  // uniform over the grid
  float* my_hi = d_hi[me.team * QROWS + me.row];
  float* my_lo = d_lo[me.team * QROWS + me.row];
#pragma unroll
  for (int t = 0; t < E; ++t)
    my_hi[me.slot + t / V * T::STRIDE + t % V] = my_lo[me.slot + t / V * T::STRIDE + t % V] = 0.f;
  __syncthreads();
  // the momentum of the next index, so that the pixel phase's last block only
  // copies it: its FP64 powers take about 5 us, here beside the projections
  // of the block's other warps
  if (blockIdx.x == 0 && tid >= Q_THREADS - W && live(slots[tid - (Q_THREADS - W)]))
    next_momentum(slots[tid - (Q_THREADS - W)]);
  const uint64_t pol = evict_first_policy();
  for (int r = 0; r < deal.rounds; ++r) {
    const int b = deal.block(a.QA, r);
    unsigned long long sums[QROWS][T::Q / 2];
    quad_sums<W, S, BF16, NZ>(a.QA, b, f, Kp, me, gather_on, pol, sums);
    const int row = b >= 0 ? __ldg(a.QA.rows + QROWS * b + me.row) : -1;
    float acc[E];
    quad_reduce<W, S>(sums, me, s_x, r & 1, acc);
    if (row < 0 || on == 0) continue;
#pragma unroll
    for (int i = 0; i < E / V; ++i) {
      const int sl = me.slot + i * T::STRIDE;
      const size_t o = (size_t)row * Kp + s0 + sl;
      float yp[V], gg[V], gm[V], wo[V], yo[V];
      if (!first) vload<V>(y_prev + o, yp);
      vload<V>(a.g + o, gg);
      vload<V>(a.gamma + o, gm);
#pragma unroll
      for (int j = 0; j < V; ++j) {
        const int t = V * i + j;
        const float y = acc[t];
        yo[j] = y;
        wo[j] = 0.f;
        if (!(on >> t & 1)) continue;
        // y~ = y + theta (y - y_prev); den = max(y~ + gamma, kappa gamma); w = (den - g)/den
        const float yt = first ? y : fmaf(s_th[sl + j], y - yp[j], y);
        float den = yt + gm[j];
        const float fl = 1e-3f * gm[j];
        if (den < fl) {
          den = fl;
          atomicAdd(&slots[sl + j].guard_hits, 1ull);
        }
        wo[j] = __fdiv_rn(den - gg[j], den);
        if (want) {
          // data term y - g ln(y + gamma) in double-float
          df yg;
          two_sum(y, gm[j], yg.hi, yg.lo);
          const df term = df_add_f(df_neg(df_mul_f(df_log(yg), gg[j])), y);
          acc_add(my_hi[sl + j], my_lo[sl + j], term.hi, term.lo);
        }
      }
      const unsigned m = on >> (V * i) & ((1u << V) - 1);
      vstore<V>(y_out + o, yo, m);
      vstore<V>(a.w + o, wo, m);
    }
  }
  if (!want) return;
  // One row of per-slot sums per virtual block, in the columns of the live
  // slots: its teams' rows in order.  An admission pass writes only the fresh
  // slots' columns.
  __syncthreads();
  constexpr int VBB = T::TB / T::TV;
  for (int q = tid; q < VBB * W; q += Q_THREADS) {
    const int s = q % W, vb = blockIdx.x * VBB + q / W;
    if (vb >= a.n_spmv_blocks || !live(slots[s])) continue;
    float h = 0.f, l = 0.f;
    for (int r = 0; r < T::TV * QROWS; ++r)
      acc_add(h, l, d_hi[q / W * T::TV * QROWS + r][s], d_lo[q / W * T::TV * QROWS + r][s]);
    a.fpartial[(size_t)vb * Kp + s0 + s] = make_float2(h, l);
  }
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
  const float lam1 = sl.lambda1, lam2 = sl.lambda2, eps = sl.eps, eps2 = square_of(eps);
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
// us one by one).  The rows of sums lie as the forward phase's; blockIdx.y takes
// the slots from y W on.
template <int W, bool BF16>
__global__ void __launch_bounds__(P_THREADS, 2) k_bobjective(BFwdArgs a) {
  using T = Team<W>;
  constexpr int E = T::E, Q = T::Q, F = Q / 4;
  __shared__ float dsum_hi[P_WARPS * T::RW][W], dsum_lo[P_WARPS * T::RW][W];
  const int lane = threadIdx.x & 31, g = lane % T::LANES / T::L;
  const int s0 = blockIdx.y * W, sl0 = s0 + owned_slot<W>(lane), Kp = a.Kp;
  const float* xl = a.f[a.bst->gstep % 3] + s0 + gathered_slot<W>(lane);
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
    const bool up2 = g >> 1;
#pragma unroll
    for (int t = 0; t < E; ++t) {
      const float sh = __shfl_xor_sync(0xffffffffu, up2 ? qh[t] : qh[E + t], 2 * T::L);
      const float sl = __shfl_xor_sync(0xffffffffu, up2 ? ql[t] : ql[E + t], 2 * T::L);
      qh[t] = up2 ? qh[E + t] : qh[t];
      ql[t] = up2 ? ql[E + t] : ql[t];
      acc_add(qh[t], ql[t], sh, sl);
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
// block adds the group sums.  Every sum runs in two parts combined in order,
// whatever the grid and the slots' number.
constexpr int OBJ_GROUPS = 64;
constexpr int OBJ_PARTS = Q_THREADS / MAXK;
__device__ void sum_rows(const float2* rows, int first, int step, int count, int Kp,
                         float (&r_hi)[Q_THREADS], float (&r_lo)[Q_THREADS]) {
  const int s = threadIdx.x % MAXK, part = threadIdx.x / MAXK;
  float h = 0.f, l = 0.f;
  if (s < Kp) {
#pragma unroll 16
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

template <int W, int S, bool BF16, int NZ>
__global__ void __launch_bounds__(Q_THREADS, Q_PER_SM) k_bpixel(BPixArgs a) {
  using T = QTeam<W, S>;
  constexpr int E = T::E, V = T::V;
  __shared__ float r_hi[Q_THREADS], r_lo[Q_THREADS];
  __shared__ float s_th[W], s_beta[W];
  __shared__ int s_frz[W];  // -1: P from f^k; 0: the same, kept as f^{K_P}; 1: P from f^{K_P}
  __shared__ float s_x[kReduceFloats<W, S>];
  __shared__ int s_last;
  BatchState* bs = a.bst;
  const int remaining = bs->remaining, G = bs->gstep;
  const QLane<W, S> me;
  const QuadDeal<W, S> deal(me, a.QT.blocks, a.n_blocks);
  deal.warm(a.QT);
  const int tid = threadIdx.x, lane = tid & 31;
  const int Kp = a.Kp, s0 = blockIdx.y * W;
  if (remaining == 0) return;  // uniform over the grid
  const float* fk = a.f[G % 3];
  const float* fkm = a.f[(G + 2) % 3];
  float* fn = a.f[(G + 1) % 3];
  // every slot's Phi(f^k): the forward phase's rows, first because these
  // blocks start first
  if (a.track && blockIdx.y == 0)
    for (int g = blockIdx.x; g < OBJ_GROUPS; g += gridDim.x) {
      sum_rows(a.fpartial, g, OBJ_GROUPS, a.n_fpartial, Kp, r_hi, r_lo);
      if (tid < Kp) a.partial[(size_t)g * Kp + tid] = make_float2(r_hi[tid], r_lo[tid]);
    }
  const SlotState* slots = a.slots + s0;
  unsigned live = 0, back = 0;  // the lane's owned slots
  bool gather_on = false;
  int freeze = 0;
#pragma unroll
  for (int t = 0; t < E; ++t) {
    const SlotState& sl = slots[me.slot + t / V * T::STRIDE + t % V];
    live |= sl.active && !sl.done ? 1u << t : 0u;
    back |= sl.rollback ? 1u << t : 0u;
    freeze |= sl.freeze_iter >= 0;
  }
#pragma unroll
  for (int t = 0; t < T::Q; ++t) {
    const SlotState& sl = slots[me.gathered() + t / 4 * T::STRIDE + t % 4];
    gather_on = gather_on || (sl.active && !sl.done);
  }
  for (int t = tid; t < W; t += Q_THREADS) {
    const SlotState& sl = slots[t];
    s_th[t] = sl.theta_hi;
    s_beta[t] = sl.beta;
    s_frz[t] = sl.freeze_iter < 0 || sl.k < sl.freeze_iter ? -1 : sl.k > sl.freeze_iter;
  }
  __syncthreads();
  const uint64_t pol = evict_first_policy();
  int bad = 0;
  for (int r = 0; r < deal.rounds; ++r) {
    const int b = deal.block(a.QT, r);
    unsigned long long sums[QROWS][T::Q / 2];
    quad_sums<W, S, BF16, NZ>(a.QT, b, a.w + s0, Kp, me, gather_on, pol, sums);
    const int j = b >= 0 ? __ldg(a.QT.rows + QROWS * b + me.row) : -1;
    float bp[E];
    quad_reduce<W, S>(sums, me, s_x, r & 1, bp);
    if (j < 0) continue;
    const float il = __ldg(a.inv_lambda + j);
#pragma unroll
    for (int i = 0; i < E / V; ++i) {
      const int sl = me.slot + i * T::STRIDE;
      const size_t o = (size_t)j * Kp + s0 + sl;
      float vk[V], vd[V], lo[V], gr[V], out[V];
      vload<V>(fk + o, vk);
      vload<V>(a.delta + o, vd);
      vload<V>(a.low + o, lo);
      vload<V>(a.gR + o, gr);
#pragma unroll
      for (int u = 0; u < V; ++u) {
        const int t = V * i + u;
        if (!(live >> t & 1)) {
          // finished or empty slot: carry the image (the previous entry when
          // the slot stopped one step back)
          out[u] = back >> t & 1 ? fkm[o + u] : vk[u];
          continue;
        }
        float pk = vk[u];
        if (freeze) {
          if (s_frz[sl + u] == 0) a.pfreeze[o + u] = vk[u];
          if (s_frz[sl + u] == 1) pk = a.pfreeze[o + u];
        }
        // f^{k+1} = max(f^k + step, 0), step = theta (f^k - f^{k-1}) - p (grad F +
        // grad R): what rounding f^{k+1} to FP32 leaves over is kept in low, and
        // the step itself is the next f^k - f^{k-1}
        const float p = s_beta[sl + u] * pk * il;
        const float step = __fmaf_rn(s_th[sl + u], vd[u], -__fmul_rn(p, bp[t] + gr[u]));
        const float full = __fadd_rn(vk[u], lo[u]);
        float xv, rest;
        two_sum(vk[u], __fadd_rn(lo[u], step), xv, rest);
        if (!isfinite(xv)) bad = 1;
        const bool pos = xv > 0.f;
        out[u] = pos ? xv : 0.f;
        vd[u] = pos ? step : -full;
        lo[u] = pos ? rest : 0.f;
      }
      const unsigned m = live >> (V * i) & ((1u << V) - 1);
      vstore<V>(fn + o, out, (1u << V) - 1);
      vstore<V>(a.delta + o, vd, m);
      vstore<V>(a.low + o, lo, m);
    }
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(&bs->flags, APPGA_FLAG_NONFINITE);
  // Finalise the step in the last block: Phi and the stopping test of every
  // live slot, then its next index and momentum; the global step advances.
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(&bs->ticket_p, 1u) == gridDim.x * gridDim.y - 1;
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
    static_assert(Q_THREADS >= MAXK, "one slot per thread");
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
// block per slice did both: 192 us for 64 slices of 256 x 256, 13 + 25 us now).
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

// Small matrices run 16 groups per block of rows (a rule on the matrix alone, so
// that a slice's result does not depend on its batch): below two teams per
// resident warp at four groups a block.  5 slots of 128 x 128 (4.1 k blocks):
// 37 us per map with four groups, 32.6 with 16.
bool many_groups(const DevQuad& M) { return M.blocks < 2 * Q_PER_SM * Q_WARPS * sm_count(); }
int virtual_blocks(const DevQuad& M, int per_sm) {
  const int tv = many_groups(M) ? 1 : 4;
  return std::min((M.blocks + tv - 1) / tv, sm_count() * per_sm);
}
// Virtual blocks of the forward phase's projection.
int fw_blocks(const BFwdArgs& a) {
  return virtual_blocks(a.QA, clamp_per_sm(a.spmv_per_sm, kSpmvPerSm));
}
// Stencil blocks per slot chunk: equal tile counts per block.
int st_blocks(const BFwdArgs& a) {
  if (a.no_stencil) return 0;
  const int tiles = ((a.n + BST_OUT - 1) / BST_OUT) * ((a.n + BST_R - 1) / BST_R);
  const int cap = sm_count() * clamp_per_sm(a.stencil_per_sm, kStencilPerSm);
  const int per = (tiles + cap - 1) / cap;
  return (tiles + per - 1) / per;
}

// Gather probe: the batched projectors' inner loop alone.  Every block of rows of
// M is reduced against the slot-minor rows of x by quad_sums and quad_reduce, dealt
// to the teams as in the projections, with no epilogue, stencil or pixel update.
template <int W, int S>
__global__ void __launch_bounds__(Q_THREADS, Q_PER_SM) k_gather_probe(DevQuad M,
                                                                      const float* __restrict__ x,
                                                                      int Kp, int nvb,
                                                                      float* __restrict__ sink) {
  __shared__ float s_x[kReduceFloats<W, S>];
  const uint64_t pol = evict_first_policy();
  const QLane<W, S> me;
  const QuadDeal<W, S> deal(me, M.blocks, nvb);
  float s = 0.f;
  for (int i = 0; i < deal.rounds; ++i) {
    float acc[QTeam<W, S>::E];
    unsigned long long sums[QROWS][QTeam<W, S>::Q / 2];
    quad_sums<W, S, false, 4>(M, deal.block(M, i), x + blockIdx.y * W, Kp, me, true, pol, sums);
    quad_reduce<W, S>(sums, me, s_x, i & 1, acc);
#pragma unroll
    for (int t = 0; t < QTeam<W, S>::E; ++t) s += acc[t];
  }
  if (s == 1.0e38f) sink[blockIdx.x] = s;  // keeps the loads; the value is never used
}

// Thread blocks of nvb virtual blocks over the slots of `width`, W at a time.
template <int W, int S>
dim3 grid_of(int nvb, int width) {
  constexpr int vbb = QTeam<W, S>::TB / QTeam<W, S>::TV;
  return dim3((nvb + vbb - 1) / vbb, width / W);
}

template <int W>
cudaError_t bforward_w(const BFwdArgs& a, cudaStream_t s) {
  if (many_groups(a.QA)) {
    void (*kern)(BFwdArgs) = a.use_bf16 ? k_bforward<W, 16, true, 4> : k_bforward<W, 16, false, 4>;
    kern<<<grid_of<W, 16>(a.n_spmv_blocks, a.width), Q_THREADS, 0, s>>>(a);
  } else {
    const bool g4 = a.gather_rows == 4;
    void (*kern)(BFwdArgs) =
        a.use_bf16 ? (g4 ? k_bforward<W, 4, true, 2> : k_bforward<W, 4, true, 4>)
                   : (g4 ? k_bforward<W, 4, false, 2> : k_bforward<W, 4, false, 4>);
    kern<<<grid_of<W, 4>(a.n_spmv_blocks, a.width), Q_THREADS, 0, s>>>(a);
  }
  return cudaGetLastError();
}
template <int W>
cudaError_t bpixel_w(const BPixArgs& a, cudaStream_t s) {
  if (many_groups(a.QT)) {
    void (*kern)(BPixArgs) = a.use_bf16 ? k_bpixel<W, 16, true, 4> : k_bpixel<W, 16, false, 4>;
    kern<<<grid_of<W, 16>(a.n_blocks, a.width), Q_THREADS, 0, s>>>(a);
  } else {
    const bool g4 = a.gather_rows == 4;
    void (*kern)(BPixArgs) =
        a.use_bf16 ? (g4 ? k_bpixel<W, 4, true, 2> : k_bpixel<W, 4, true, 4>)
                   : (g4 ? k_bpixel<W, 4, false, 2> : k_bpixel<W, 4, false, 4>);
    kern<<<grid_of<W, 4>(a.n_blocks, a.width), Q_THREADS, 0, s>>>(a);
  }
  return cudaGetLastError();
}
template <int W>
cudaError_t probe_w(const DevQuad& M, const float* x, int Kp, float* sink, int per_sm,
                    cudaStream_t s) {
  const int nvb = virtual_blocks(M, per_sm);
  if (many_groups(M))
    k_gather_probe<W, 16><<<grid_of<W, 16>(nvb, Kp), Q_THREADS, 0, s>>>(M, x, Kp, nvb, sink);
  else
    k_gather_probe<W, 4><<<grid_of<W, 4>(nvb, Kp), Q_THREADS, 0, s>>>(M, x, Kp, nvb, sink);
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
    case 64:
    case 128: return bforward_w<64>(a, s);
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
  const dim3 grid((a.n_spmv_blocks + Team<W>::RW - 1) / Team<W>::RW, a.width / W);
  if (a.use_bf16)
    k_bobjective<W, true><<<grid, P_THREADS, 0, s>>>(a);
  else
    k_bobjective<W, false><<<grid, P_THREADS, 0, s>>>(a);
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_bobjective(const BFwdArgs& a0, int K, double* out, cudaStream_t s) {
  cudaError_t e = ensure_tables();
  if (e != cudaSuccess) return e;
  BFwdArgs a = a0;
  a.mode = 3;
  a.track = 1;
  a.n_spmv_blocks =
      std::min((a.A.rows + P_WARPS - 1) / P_WARPS, sm_count() * kObjectivePerSm);
  switch (a.width) {
    case 8: e = bobjective_w<8>(a, s); break;
    case 16: e = bobjective_w<16>(a, s); break;
    case 32: e = bobjective_w<32>(a, s); break;
    case 64:
    case 128: e = bobjective_w<64>(a, s); break;
    default: e = cudaErrorInvalidValue;
  }
  const int nst = st_blocks(a);
  if (e == cudaSuccess && nst > 0) {
    k_bstencil<<<dim3(nst, a.width / BST_S), B_THREADS, 0, s>>>(a);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return e;
  k_sum_columns<<<K, 256, 0, s>>>(a.fpartial, a.n_spmv_blocks, nst, a.Kp, out);
  return cudaGetLastError();
}

cudaError_t launch_gather_probe(const DevQuad& M, const float* x, int Kp, float* sink,
                                int blocks_per_sm, cudaStream_t s) {
  if (blocks_per_sm < 1 || blocks_per_sm > kMaxPerSm) return cudaErrorInvalidValue;
  switch (Kp) {
    case 32: return probe_w<32>(M, x, Kp, sink, blocks_per_sm, s);
    case 64:
    case 128: return probe_w<64>(M, x, Kp, sink, blocks_per_sm, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_bpixel(const BPixArgs& a0, cudaStream_t s) {
  BPixArgs a = a0;
  a.n_blocks = virtual_blocks(a.QT, clamp_per_sm(a.blocks_per_sm, kPixelPerSm));
  switch (a.width) {
    case 8: return bpixel_w<8>(a, s);
    case 16: return bpixel_w<16>(a, s);
    case 32: return bpixel_w<32>(a, s);
    case 64:
    case 128: return bpixel_w<64>(a, s);
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
