// Device structures and launchers of the batched (multi-slice) kernels.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "appga_internal.h"

namespace appga {

// Per-slot device state: iteration index, momentum, objective, stop flag and
// the slot's model parameters.  Slots are independent problems sharing A.
struct SlotState {
  int32_t k;          // index of the slot's current iterate
  int32_t k0;         // first index of the slot's run
  int32_t k_last;     // last step index to run
  int32_t done;       // finished (iteration cap or stopping test)
  int32_t result_k;   // index of the slot's result
  int32_t stopped_early;
  int32_t active;     // the slot holds a problem
  int32_t freeze_iter;
  int32_t momentum;
  int32_t fresh;      // just admitted: f^{k-1} = f^k, needs its first forward phase
  int32_t phi_k;      // iterate index whose objective is in phi_cur (-1: none)
  int32_t rollback;   // stopped one step back: the result is the previous ring entry
  float theta_hi, theta_lo;  // theta_k as a double-float pair
  float lambda1, lambda2, eps, beta;
  double theta, t_cur, phi_cur, phi_prev;
  double theta_next, t_next;  // momentum of index k + 1 (set by the forward phase of k)
  double omega, a, b, rel_tol;
  unsigned long long guard_hits;
};

struct BatchState {
  int32_t gstep;      // global step: ring slot of the current iterates
  int32_t remaining;  // live slots
  int32_t flags;
  int32_t phi_tot_k;  // volume mode: iterate index of phi_tot_cur (-1: none)
  unsigned int ticket_r, ticket_p, ticket_aux, pad2;
  double phi_tot_cur, phi_tot_prev;  // volume mode: objective of the whole volume
};

struct BFwdArgs {
  DevQuad QA;
  DevCSR A;       // the objective's double-float projections
  int32_t n;
  int32_t Kp;     // row stride of the slot-minor arrays
  int32_t width;  // slots worked on: 8, 16, 32, 64 or 128, every live slot below it
  int32_t mode;   // 0: solver step; 1: first forward phase of a run (f^{k-1} = f^k);
                  // 2: first forward phase of the fresh slots only (admission);
                  // 3: objective of every active slot's result
  int32_t track;
  int32_t use_bf16;
  int32_t n_spmv_blocks;  // virtual blocks of the projection, set by the launcher
  int32_t spmv_per_sm;    // virtual blocks per SM (0: default); tuned by the autotuner
  int32_t stencil_per_sm; // stencil blocks per SM (0: default)
  int32_t no_stencil;     // volume mode: the 3-D stencil takes the 2-D one's place
  int32_t gather_rows;    // image rows a lane gathers per step: 8 (0: default) or 4; tuned
  float* f[3];
  const float* delta;  // f^k - f^{k-1}, and what rounding f^k to FP32 left over
  const float* low;
  float* y[2];
  float* w;
  const float* g;
  const float* gamma;
  float* gR;
  SlotState* slots;
  BatchState* bst;
  float2* fpartial;  // per-slot objective partials, one row of Kp per block
};

struct BPixArgs {
  DevQuad QT;
  int32_t n;
  int32_t Kp;             // row stride of the slot-minor arrays
  int32_t width;          // slots worked on (as BFwdArgs)
  int32_t use_bf16;
  int32_t n_blocks;       // virtual blocks, set by the launcher
  int32_t blocks_per_sm;  // 0: default; tuned by the autotuner
  int32_t gather_rows;    // weight rows a lane gathers per step: 8 (0: default) or 4; tuned
  float* f[3];
  float* delta;  // as BFwdArgs, of the current step, replaced by the next step's
  float* low;
  const float* w;
  const float* gR;
  const float* inv_lambda;
  float* pfreeze;
  SlotState* slots;
  BatchState* bst;
  float2* partial;  // group sums of the objective partials
  // objective partials left by the forward phase of the same step (track):
  // reduced here, where the stopping test runs
  const float2* fpartial;
  int32_t n_fpartial;
  int32_t track;
  int32_t joint;  // volume mode: one stopping test on the sum of the slots' objectives
};

// 3-D SHOITV stencil (kernels_vol.cu) on slice-major volumes: voxel
// (z, r, c) at z n^2 + r n + c.  Solver mode (bst != null): f^k and f^{k-1}
// are the slice-major ring entries of the current step (f[G % 3] and
// f[(G + 2) % 3]), theta, lambda and eps come from slot z; stand-alone mode:
// f[0] is the volume, f~ = f, lam1/lam2/eps as given.
struct Vol3Args {
  int32_t n, nz;
  const float* f[3];
  const SlotState* slots;
  const BatchState* bst;
  float lam1, lam2, eps;
  int32_t want_reg;       // also the regulariser at f^k: one row of pstride
  int32_t pstride;        // per-slice double-float sums per block in partial
  int32_t pad;
  float* gR;              // out: B^T grad phi~(B f~), slice-major
  float2* partial;        // out (want_reg): stencil3d_grid rows of pstride
};
int stencil3d_max_slices();
int stencil3d_grid(int n, int nz);
cudaError_t launch_stencil3d(const Vol3Args& a, cudaStream_t s);
// *out = sum of rows x cols double-float pairs (row stride pstride), in FP64
cudaError_t launch_sum_pairs(const float2* p, int rows, int cols, int pstride, double* out,
                             cudaStream_t s);
// Volume mode: the current ring entry (bst->gstep) of the slot-minor iterate
// ring [d][Kp] into the slice-major ring [nz][d] (every entry if all != 0),
// and a slice-major gradient [nz][d] into the slot-minor [d][Kp].  Both do
// nothing once no slot is live.
cudaError_t launch_slots_to_slices(float* const* slot_ring, float* const* slice_ring, int d,
                                   int Kp, int nz, const BatchState* bst, int all,
                                   cudaStream_t s);
cudaError_t launch_slices_to_slots(const float* in, float* out, int d, int Kp, int nz,
                                   const BatchState* bst, cudaStream_t s);

int batch_max_blocks();
// Rows of objective partials a forward phase with these arguments leaves
// (its projection's virtual blocks, then its stencil blocks).
int bforward_grid(const BFwdArgs& a);
// Slots whose result sits one ring entry back (stopped by the test in the
// last pixel phase): copy it into the current entry and clear the mark.
cudaError_t launch_resolve_rollback(const BFwdArgs& a, cudaStream_t s);
cudaError_t launch_bforward(const BFwdArgs& a, cudaStream_t s);
// The forward phase's 2-D stencil, on the same arguments; independent of
// launch_bforward (they may overlap).
cudaError_t launch_bstencil(const BFwdArgs& a, cudaStream_t s);
// Objective of the results in the current ring entry, slots 0 .. K - 1: the
// data term of slot s into out[2 s], its regulariser into out[2 s + 1] (0 with
// a.no_stencil).  Uses the objective rows (fpartial) and gR as scratch.
cudaError_t launch_bobjective(const BFwdArgs& a, int K, double* out, cudaStream_t s);
// The batched projectors' inner loop alone over M (rows reduced against the
// Kp-wide rows of x, [cols][Kp]; no epilogue) with blocks_per_sm (1..16)
// blocks per SM; sink: at least (SMs x 16) floats, written only in a case
// that does not arise.
cudaError_t launch_gather_probe(const DevQuad& M, const float* x, int Kp, float* sink,
                                int blocks_per_sm, cudaStream_t s);
// Slots the kernels work on for K slices: the narrowest of 8, 16, 32, 64 and
// 128 that holds them.
inline int slot_width(int K) {
  int w = 8;
  while (w < K) w *= 2;
  return w;
}
cudaError_t launch_bpixel(const BPixArgs& a, cudaStream_t s);
// Slot lists: where `ids` is given, slice k goes to slot ids[k] (a device
// array of K ints); otherwise to slot s0 + k.
cudaError_t launch_binit_momentum(SlotState* slots, int Kp, bool only_fresh, cudaStream_t s);
// (fill: value of the padding slots when ids == NULL; flag, may be NULL: set
// to 1 if a value is not finite, negative or, with positive, zero)
cudaError_t launch_to_slot_minor(const float* in, int K, int len, float* out, int Kp, int s0,
                                 const int* ids, cudaStream_t s, float fill = 0.f,
                                 bool positive = false, int* flag = nullptr);
// images (a.n^2 pixels) of K slots of the current ring entry, slice-major
cudaError_t launch_from_slot_minor(const BFwdArgs& a, int K, int s0, const int* ids, float* out,
                                   cudaStream_t s);
cudaError_t launch_fill_slots(float* out, int len, int Kp, int s0, int s1, float v, cudaStream_t s);
cudaError_t launch_binit_image(const float* g, const float* gamma, int m, int n, int n_angles,
                               long long npfov, int K, int Kp, int s0, const int* ids,
                               float2* scratch, float* f_cur, float* f_prev, float* delta,
                               float* low, cudaStream_t s);

}  // namespace appga
