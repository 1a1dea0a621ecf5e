// Device arguments and launchers of the AFPPA kernels (kernels_afppa.cu).
#pragma once

#include <cuda_runtime.h>

#include "appga_internal.h"

namespace appga {

struct DualArgs {
  int32_t n;               // image side
  float lambda1, lambda2;  // ball radii of the dual groups
  const float* f[3];       // iterate ring
  float* b[3];             // first-order dual ring, [2][d] (field-major)
  float* c[3];             // second-order dual ring, [4][d]
  float* gR;               // out: B1^T b~ + B2^T c~ for the next pixel phase
  SolverState* st;         // k (the step's index), p_max; receives rho1, rho2
  const ThetaEntry* theta_tab;  // theta_{k0+i} of the run
};

// Result of a run: the ring entries of f^{r}, b^{r}, c^{r} (r = st->result_k) to
// f_out, b_out, c_out (the duals may be NULL), and ||f^{r} - f^{r-1}||^2,
// ||f^{r}||^2 into norms[2]; nothing if the inputs failed the check.  partial:
// scratch of kAfppaResultBlocks float4.
constexpr int kAfppaResultBlocks = 128;
struct AfppaResultArgs {
  int32_t d;
  const float* f[3];
  const float* b[3];
  const float* c[3];
  const SolverState* st;
  float *f_out, *b_out, *c_out;
  float4* partial;
  double* norms;
};

cudaError_t launch_afppa_dual(const DualArgs& a, cudaStream_t s);
cudaError_t launch_afppa_result(const AfppaResultArgs& a, cudaStream_t s);

}  // namespace appga
