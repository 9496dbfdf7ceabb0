// simt_project.h - fused snapshot difference + multi-mode projection in float and double on
// the CUDA cores: the projection of Eqs. 2.15/2.16 without reduced-precision operands.
#pragma once
#include <string>

#include "kernels.h"

namespace tdb {

struct SpPlan {
  void* z1p = nullptr;                // [tiles along i1][slices][r1][N2] partial dV x_1 A_1^T
  void* z2p = nullptr;                // [tiles along i2][slices][r2][N1] partial dV x_2 A_2^T
  double* wsl = nullptr;              // product of the weights of modes >= 3, per slice
  double* npart = nullptr;            // ||dV||_W^2 per warp of every CTA
  void* fpart = nullptr;              // split partials of the finishing contraction
  size_t fpart_cap = 0;               // values
  void* wrest = nullptr;              // W = Z1 x_2 A_2^T of four modes (r1 x r2 x N3 x N4)
};

// Whether the pass is the faster way for tensors of these sizes.
template <typename T>
bool sp_worth(int p, const int64_t* N);
// Whether sp_project takes these ranks (r_3 r_4 of four modes at most 128).
bool sp_supported(int p, const int* r);
// The slice weights, kept for the context's life, and the buffers of a pass, free between passes.
void sp_carve_weights(SpPlan& plan, Carver& cv, int p, const int64_t* N);
template <typename T>
void sp_carve_pass(SpPlan& plan, Carver& cv, int p, const int64_t* N, const int* cap);
// The slice weights, once per context (before any capture).
void sp_prepare(SpPlan& plan, int p, const int64_t* N, const double* const* w, cudaStream_t s);
// Y_n of dV = dscale (Vn - Vp) (Eqs. 2.15, 2.16; dscale a power of two) and ||dV||_W^2 into
// *dv2; dS = Y_2 x_2 A_2^T is left to the update kernel.  A: weighted bases (N_n x r_n);
// w: mode weights; Z1: r1 x N2 x S scratch.  A non-finite difference sets kFlagNonFinite.
// evm (nullable): two events around the main kernel.
template <typename T>
tdb_status sp_project(SpPlan& plan, const T* Vn, const T* Vp, int p, const int64_t* N, const int* r,
                      const void* const* A, const double* const* w, T* Z1, T* const* Y, double* dv2, unsigned* flags,
                      cudaStream_t s, cudaEvent_t* evm, std::string& err, T dscale);

}  // namespace tdb
