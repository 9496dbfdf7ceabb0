// k_eig.cu - the weighted mode Grams of the float compute types (Sec. 2.3 last paragraph,
// Sec. 2.5):
//     C_n = W_n^{1/2} V_(n) W_{-n} V_(n)^T W_n^{1/2}
// formed as Vw_(n) Vw_(n)^T with Vw = V scaled by sqrt(w_1 ... w_p) once.
//
// Precision: products in float, 32-column chunk sums in float, chunks accumulated
// as float-float pairs (TwoSum), so the Gram carries the float rounding of the
// chunk sums and nothing coarser.
#include "common.cuh"
#include "kernels.h"

namespace tdb {

namespace {

constexpr int SY_T = 64;          // Gram output tile
constexpr int SY_K = 32;          // columns per chunk

__device__ __forceinline__ void two_sum(float& hi, float& lo, float x) {
  const float s = hi + x;
  const float bb = s - hi;
  const float err = (hi - (s - bb)) + (x - bb);
  hi = s;
  lo += err;
}

}  // namespace

// ---------------------------------------------------------------------------
// Vw = V * sqrt(w_1[i_1] ... w_p[i_p])   (ws[n] = sqrt(w_n) in float)
// ---------------------------------------------------------------------------
struct SqrtWeights {
  int p;
  int N[kMaxModes];
  const float* ws[kMaxModes];
};

__global__ void k_weight_data(const float* __restrict__ V, SqrtWeights sw, int S, float* __restrict__ Vw) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < S; e += gridDim.x * blockDim.x) {
    int rem = e;
    float f = 1.f;
    for (int n = 0; n < sw.p; ++n) {
      const int i = rem % sw.N[n];
      rem /= sw.N[n];
      f *= sw.ws[n][i];
    }
    Vw[e] = V[e] * f;
  }
}

__global__ void k_sqrt_weights(const double* __restrict__ w, int n, float* __restrict__ ws) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) ws[i] = (float)sqrt(w[i]);
}

// ---------------------------------------------------------------------------
// Gram tiles: blockIdx.x = upper tile pair (ti <= tj) of 64 x 64, blockIdx.y =
// column slice.  256 threads, 4 x 4 outputs each.  Column c of Vw_(n) is (l, q):
// Vw[l + L (i + N q)].
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_syrk_partial(const float* __restrict__ Vw, int64_t L, int64_t Nn, int64_t Q,
                                                      int ntile, int ksplit, double* __restrict__ part) {
  int t = blockIdx.x, ti = 0;
  while (t >= ntile - ti) { t -= ntile - ti; ++ti; }
  const int tj = ti + t;
  const bool diag = (ti == tj);
  const int64_t i0 = (int64_t)ti * SY_T, j0 = (int64_t)tj * SY_T;
  const int64_t ncol = L * Q;
  const int64_t c0 = ncol * blockIdx.y / ksplit, c1 = ncol * (blockIdx.y + 1) / ksplit;
  __shared__ __align__(16) float As[SY_K][SY_T + 4];
  __shared__ __align__(16) float Bs[SY_K][SY_T + 4];
  const int tid = threadIdx.x;
  const int tr = tid & 15, tc = tid >> 4;       // output rows tr*4.., columns tc*4..
  const bool rows_fast = (L == 1);
  // load mapping: 8 elements per panel per thread.  With L == 1 the lanes run along
  // rows (contiguous) and column c is q = c; otherwise the lanes run along columns
  // (l contiguous) and each thread keeps its column's (l, q), advanced by 32 per chunk.
  const int ccol = tid & 31;
  int64_t lcur = 0, qcur = 0;
  if (!rows_fast) { lcur = (c0 + ccol) % L; qcur = (c0 + ccol) / L; }
  auto load = [&](int64_t cb, float* ra, float* rb) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      int ri;
      int64_t c, l, q;
      if (rows_fast) { ri = tid & 63; c = cb + (tid >> 6) + 4 * u; l = 0; q = c; }
      else { ri = (tid >> 5) + 8 * u; c = cb + ccol; l = lcur; q = qcur; }
      float va = 0.f, vb = 0.f;
      if (c < c1) {
        const int64_t ia = i0 + ri, ib = j0 + ri;
        if (ia < Nn) va = Vw[l + L * (ia + Nn * q)];
        if (!diag && ib < Nn) vb = Vw[l + L * (ib + Nn * q)];
      }
      ra[u] = va;
      rb[u] = vb;
    }
    if (!rows_fast) {
      lcur += SY_K;
      while (lcur >= L) { lcur -= L; ++qcur; }
    }
  };
  auto store = [&](const float* ra, const float* rb) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      int ri, cc;
      if (rows_fast) { ri = tid & 63; cc = (tid >> 6) + 4 * u; }
      else { cc = ccol; ri = (tid >> 5) + 8 * u; }
      As[cc][ri] = ra[u];
      if (!diag) Bs[cc][ri] = rb[u];
    }
  };
  float hi[16], lo[16];
#pragma unroll
  for (int x = 0; x < 16; ++x) { hi[x] = 0.f; lo[x] = 0.f; }
  float ra[8], rb[8];
  load(c0, ra, rb);
  for (int64_t cb = c0; cb < c1; cb += SY_K) {
    __syncthreads();
    store(ra, rb);
    __syncthreads();
    if (cb + SY_K < c1) load(cb + SY_K, ra, rb);
    const float (*Bp)[SY_T + 4] = diag ? As : Bs;
    float acc[16];
#pragma unroll
    for (int x = 0; x < 16; ++x) acc[x] = 0.f;
#pragma unroll 4
    for (int k = 0; k < SY_K; ++k) {
      const float4 a = *reinterpret_cast<const float4*>(&As[k][tr * 4]);
      const float4 b = *reinterpret_cast<const float4*>(&Bp[k][tc * 4]);
      const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) acc[x * 4 + y] = fmaf(av[x], bv[y], acc[x * 4 + y]);
    }
#pragma unroll
    for (int x = 0; x < 16; ++x) two_sum(hi[x], lo[x], acc[x]);
  }
  double* out = part + ((int64_t)blockIdx.x * ksplit + blockIdx.y) * SY_T * SY_T;
#pragma unroll
  for (int x = 0; x < 4; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y)
      out[(tr * 4 + x) + SY_T * (tc * 4 + y)] = (double)hi[x * 4 + y] + (double)lo[x * 4 + y];
}

// Sum the slices: C64, full n x n.
__global__ void k_syrk_finish(int64_t Nn, int ntile, int ksplit, const double* __restrict__ part,
                              double* __restrict__ C64) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < Nn * Nn; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e % Nn, j = e / Nn;
    const int64_t a = i <= j ? i : j, b = i <= j ? j : i;
    const int ti = (int)(a / SY_T), tj = (int)(b / SY_T);
    const int pair = ti * ntile - ti * (ti - 1) / 2 + (tj - ti);
    int x = (int)(a % SY_T), y = (int)(b % SY_T);
    if (ti == tj && x > y) { const int t = x; x = y; y = t; }
    double s = 0.0;
    const double* src = part + (int64_t)pair * ksplit * SY_T * SY_T + x + SY_T * y;
#pragma unroll 8
    for (int k = 0; k < ksplit; ++k) s += src[(int64_t)k * SY_T * SY_T];
    C64[e] = s;
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
void launch_sqrt_weights(const double* w, int n, float* ws, cudaStream_t s) {
  k_sqrt_weights<<<std::max(1, std::min((n + 255) / 256, 64)), 256, 0, s>>>(w, n, ws);
  count_launch();
}

void launch_weight_data(const float* V, int p, const int64_t* N, const float* const* ws, int64_t S, float* Vw,
                        cudaStream_t s) {
  SqrtWeights sw;
  sw.p = p;
  for (int n = 0; n < kMaxModes; ++n) {
    sw.N[n] = n < p ? (int)N[n] : 1;
    sw.ws[n] = n < p ? ws[n] : nullptr;
  }
  const int blocks = (int)std::min<int64_t>((S + 255) / 256, 152 * 8);
  k_weight_data<<<blocks, 256, 0, s>>>(V, sw, (int)S, Vw);
  count_launch();
}

void launch_gram_weighted(const float* Vw, int64_t L, int64_t Nn, int64_t Q, double* part, size_t part_cap, double* C64,
                          cudaStream_t s) {
  const int ntile = (int)((Nn + SY_T - 1) / SY_T);
  const int npair = ntile * (ntile + 1) / 2;
  const int64_t ncol = L * Q;
  int ksplit = (int)std::max<int64_t>(1, std::min<int64_t>((152 + npair - 1) / npair, (ncol + 127) / 128));
  while ((size_t)npair * ksplit * SY_T * SY_T > part_cap && ksplit > 1) --ksplit;
  k_syrk_partial<<<dim3(npair, ksplit), 256, 0, s>>>(Vw, L, Nn, Q, ntile, ksplit, part);
  count_launch();
  const int blocks = (int)std::min<int64_t>((Nn * Nn + 255) / 256, 1024);
  k_syrk_finish<<<blocks, 256, 0, s>>>(Nn, ntile, ksplit, part, C64);
  count_launch();
}

}  // namespace tdb
