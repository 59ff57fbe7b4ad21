// FP64 iterative-refinement helpers of the Wiener filter (see wf_refine.cu).
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

namespace wf {

struct RefineArgs {
  int H, W;
  const float* d;
  const float* Nd;       // noise variance (observed pixels)
  const uint8_t* mask;
  const float* A;        // diagonal pixel response of d = A s + n, or null for A = I
  const float* Pk;       // [H][W/2+1]
  const float* s;        // current FP32 iterate [H][W]
  const float2* dn;      // Wiener-filter pixel table (d, 1/N_bar), [W][H] or, with row_major, [H][W]
  float2* rtab;          // out: correction right-hand-side table (r, 1/N_bar) in the same order
  int row_major;
  double* rnorm;         // out (refine_residual): ||S r||^2
  double* bnorm;         // out (refine_bnorm): ||S N^-1 d||^2
  void* scratch;         // refine_scratch_bytes(H, W)
};

size_t refine_scratch_bytes(int H, int W);
cudaError_t refine_bnorm(const RefineArgs& a, cudaStream_t st);
// the norm of the current iterate's residual; leaves the row transforms of s in scratch
cudaError_t refine_residual(const RefineArgs& a, cudaStream_t st);
// after refine_residual: the right-hand side r = A N^-1 (d - A s) - S^-1 s of the correction solve into rtab
cudaError_t refine_correction(const RefineArgs& a, cudaStream_t st);
cudaError_t refine_update(int n, float* s, const float* e, cudaStream_t st);
// (kappa_E, kappa_B) of shear pairs [fields][2][H][W] by the inverse Kaiser-Squires rotation; scratch: fields H W
// double2
cudaError_t shear_to_convergence_f64(const float* gamma, int fields, int H, int W, float* kappa, void* scratch,
                                     cudaStream_t st);
// spin-2 Wiener-filter residual in FP64: out[0] = ||g + S N^-1 (g - d)||^2 (g = (g1, g2), the shear
// covariance S of the E/B spectra), out[1] = ||S N^-1 d||^2 (when with_b); scratch: 2 H W double2; H <= 512
cudaError_t spin2_residual_f64(const float* g, const float* d1, const float* d2, const float* N1, const float* N2,
                               const uint8_t* mask, const float* PE, const float* PB, int H, int W, bool with_b,
                               double* out, void* scratch, cudaStream_t st);
// out = S v = U^dagger diag(P) U v in FP64 (rounded once to float); scratch: H W double2
cudaError_t apply_S_f64(const float* v, const float* Pk, int H, int W, float* out, void* scratch, cudaStream_t st);

}  // namespace wf
