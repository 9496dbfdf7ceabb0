// small_dev.cuh - shared-memory dense kernels used inside single CTAs:
// Cholesky and triangular inverse.
#pragma once
#include "common.cuh"
#include "fastrcp.cuh"

namespace tdb {

// Cholesky of the SPD matrix S (r x r, shared, leading dim lda) in place: lower
// factor L with S = L L^T.  Returns false if a pivot is not positive.
template <typename T>
__device__ __forceinline__ bool chol_smem_t(T* S, int lda, int r, bool* ok_sh) {
  if (threadIdx.x == 0) *ok_sh = true;
  __syncthreads();
  __shared__ T inv_dk;
  for (int k = 0; k < r; ++k) {
    if (threadIdx.x == 0) {
      T d = S[k + lda * k];
      if (!(d > T(0))) { *ok_sh = false; d = T(1); }
      if constexpr (sizeof(T) == 8) {
        const double y = drsqrt(d);     // one reciprocal square root per pivot (Newton-refined)
        S[k + lda * k] = d * y;
        inv_dk = y;
      } else {
        const T sd = sqrt(d);
        S[k + lda * k] = sd;
        inv_dk = T(1) / sd;
      }
    }
    __syncthreads();
    const T ik = inv_dk;
    for (int i = k + 1 + threadIdx.x; i < r; i += blockDim.x) S[i + lda * k] *= ik;
    __syncthreads();
    for (int e = threadIdx.x; e < (r - k - 1) * (r - k - 1); e += blockDim.x) {
      int i = k + 1 + e % (r - k - 1), j = k + 1 + e / (r - k - 1);
      if (j <= i) S[i + lda * j] -= S[i + lda * k] * S[j + lda * k];
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < r * r; e += blockDim.x) {
    int i = e % r, j = e / r;
    if (j > i) S[i + lda * j] = T(0);
  }
  __syncthreads();
  return *ok_sh;
}
__device__ __forceinline__ bool chol_smem(double* S, int lda, int r, bool* ok_sh) { return chol_smem_t<double>(S, lda, r, ok_sh); }

// Inverse of the lower-triangular L (shared) into Li (shared): column j solves L x = e_j.
template <typename T>
__device__ __forceinline__ void trinv_lower_smem_t(const T* L, T* Li, int lda, int r) {
  for (int j = threadIdx.x; j < r; j += blockDim.x) {
    for (int i = 0; i < r; ++i) {
      if (i < j) { Li[i + lda * j] = T(0); continue; }
      T s = (i == j) ? T(1) : T(0);
      for (int k = j; k < i; ++k) s -= L[i + lda * k] * Li[k + lda * j];
      Li[i + lda * j] = s / L[i + lda * i];
    }
  }
  __syncthreads();
}
__device__ __forceinline__ void trinv_lower_smem(const double* L, double* Li, int lda, int r) {
  trinv_lower_smem_t<double>(L, Li, lda, r);
}

}  // namespace tdb
