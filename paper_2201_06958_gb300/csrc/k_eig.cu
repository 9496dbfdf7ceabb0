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

constexpr int SY_T = 64;          // Gram output tile of modes of up to 64 points
constexpr int SY_B = 128;         // of longer ones
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

// A warp per mode-1 column: the other modes' factors once per column, 16-byte accesses where
// the columns allow them.  Bound: HBM, one read and one write of S floats (256 x 128 x 512:
// 20 us; forming every element's index from its offset took 96 us).
__global__ void __launch_bounds__(256) k_weight_data(const float* __restrict__ V, SqrtWeights sw, unsigned ncol, int vec,
                                                     float* __restrict__ Vw) {
  const int lane = threadIdx.x & 31;
  const unsigned N1 = (unsigned)sw.N[0], nw = gridDim.x * (blockDim.x >> 5);
  for (unsigned c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); c < ncol; c += nw) {
    float f[kMaxModes - 1];
    unsigned rem = c;
#pragma unroll
    for (int n = 1; n < kMaxModes; ++n) {
      f[n - 1] = 1.f;
      if (n < sw.p) {
        f[n - 1] = sw.ws[n][rem % (unsigned)sw.N[n]];
        rem /= (unsigned)sw.N[n];
      }
    }
    const float* v = V + (size_t)N1 * c;
    float* o = Vw + (size_t)N1 * c;
    auto fac = [&](float w) { return ((w * f[0]) * f[1]) * f[2]; };
    if (vec) {
      for (unsigned i = 4 * lane; i < N1; i += 128) {
        const float4 x = __ldcs((const float4*)(v + i)), w = __ldg((const float4*)(sw.ws[0] + i));
        *(float4*)(o + i) = make_float4(x.x * fac(w.x), x.y * fac(w.y), x.z * fac(w.z), x.w * fac(w.w));
      }
    } else {
      for (unsigned i = lane; i < N1; i += 32) o[i] = __ldcs(v + i) * fac(__ldg(sw.ws[0] + i));
    }
  }
}

__global__ void k_sqrt_weights(const double* __restrict__ w, int n, float* __restrict__ ws) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) ws[i] = (float)sqrt(w[i]);
}

// ---------------------------------------------------------------------------
// Gram tiles of modes of up to 64 points: blockIdx.x = upper tile pair (ti <= tj) of 64 x 64, blockIdx.y =
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

// The same with 128 x 128 tiles and 8 x 8 outputs a thread (rows 4 tr .. and 64 + 4 tr ..,
// columns 4 tc .. and 64 + 4 tc ..): a quarter of the shared-memory reads per product.  The
// next chunk of 32 columns arrives by cp.async in a second buffer (no registers held: acc, hi
// and lo take 192).  Rows of a column live in 16-byte granules, granule g of column k at
// g ^ (k & 7), so that either loading writes without bank conflicts.  On a diagonal tile the
// lower left quarter is left out (the finish reads the upper triangle).  Bound: FP32 issue at
// eight warps per SM (paired multiply-adds do not help: 0.82 ms).  256 x 128 x 512: the three
// modes 0.75 ms, with 64 x 64 tiles 1.52 ms.
__device__ __forceinline__ void sy_cp4(float* dst, const float* src, bool in) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(in ? 4 : 0) : "memory");
}
__device__ __forceinline__ void sy_cp16(float* dst, const float* src, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(in ? 16 : 0) : "memory");
}
constexpr size_t kSyrkBigSmem = 2 * 2 * sizeof(float) * SY_K * SY_B;
__global__ void __launch_bounds__(256, 1) k_syrk_big(const float* __restrict__ Vw, int64_t L, int64_t Nn, int64_t Q,
                                                     int ntile, int ksplit, double* __restrict__ part) {
  int t = blockIdx.x, ti = 0;
  while (t >= ntile - ti) { t -= ntile - ti; ++ti; }
  const int tj = ti + t;
  const bool diag = (ti == tj);
  const int64_t ncol = L * Q;
  const int64_t c0 = ncol * blockIdx.y / ksplit, c1 = ncol * (blockIdx.y + 1) / ksplit;
  extern __shared__ __align__(16) float sy_sm[];            // [buffer][A, B][SY_K][SY_B]
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int tr = tid & 15, tc = tid >> 4;
  const bool rows_fast = (L == 1);
  const bool vec = rows_fast && (Nn & 3) == 0;
  // columns fast: lanes take 8 columns x 4 rows (32-byte runs); this thread's column of group
  // kg (of 8) is cb + 8 kg + (lane & 7), its element offset at row 0 kept with its l
  int lc[4];
  int64_t oc[4];
#pragma unroll
  for (int kg = 0; kg < 4; ++kg) {
    const int64_t c = c0 + 8 * kg + (lane & 7);
    lc[kg] = rows_fast ? 0 : (int)(c % L);
    oc[kg] = rows_fast ? 0 : c % L + L * Nn * (c / L);
  }
  const int64_t wrap = L * (Nn - 1);                        // from the end of one l run to the next q's
  auto issue = [&](int64_t cb, int buf) {
    float* A = sy_sm + buf * 2 * SY_K * SY_B;
    float* Bm = A + SY_K * SY_B;
    if (rows_fast) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int k = w + 8 * u, at = k * SY_B + 4 * (lane ^ (k & 7));   // a column per warp and u
        const int64_t c = cb + k;
        const int ia = ti * SY_B + 4 * lane, ib = tj * SY_B + 4 * lane;
        const float* src = Vw + Nn * (c < c1 ? c : c0);
        if (vec) {
          sy_cp16(A + at, src + (ia < Nn ? ia : 0), c < c1 && ia < Nn);
          if (!diag) sy_cp16(Bm + at, src + (ib < Nn ? ib : 0), c < c1 && ib < Nn);
        } else {
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            sy_cp4(A + at + x, src + (ia + x < Nn ? ia + x : 0), c < c1 && ia + x < Nn);
            if (!diag) sy_cp4(Bm + at + x, src + (ib + x < Nn ? ib + x : 0), c < c1 && ib + x < Nn);
          }
        }
      }
    } else {
#pragma unroll
      for (int kg = 0; kg < 4; ++kg) {
        const int kk = 8 * kg + (lane & 7);
        const bool in = cb + kk < c1;
        const float* src = Vw + (in ? oc[kg] : 0);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int g = w + 8 * u, row = 4 * g + (lane >> 3), at = kk * SY_B + 4 * (g ^ (kk & 7)) + (lane >> 3);
          const int ia = ti * SY_B + row, ib = tj * SY_B + row;
          sy_cp4(A + at, src + (ia < Nn ? L * ia : 0), in && ia < Nn);
          if (!diag) sy_cp4(Bm + at, src + (ib < Nn ? L * ib : 0), in && ib < Nn);
        }
        lc[kg] += SY_K;
        oc[kg] += SY_K;
        while (lc[kg] >= L) { lc[kg] -= (int)L; oc[kg] += wrap; }
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float hi[64], lo[64];
#pragma unroll
  for (int x = 0; x < 64; ++x) { hi[x] = 0.f; lo[x] = 0.f; }
  issue(c0, 0);
  int buf = 0;
  for (int64_t cb = c0; cb < c1; cb += SY_K, buf ^= 1) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();                                        // this chunk is in; the other buffer is free
    if (cb + SY_K < c1) issue(cb + SY_K, buf ^ 1);
    const float* A = sy_sm + buf * 2 * SY_K * SY_B;
    const float* Bm = diag ? A : A + SY_K * SY_B;
    float acc[64];
#pragma unroll
    for (int x = 0; x < 64; ++x) acc[x] = 0.f;
#pragma unroll 4
    for (int k = 0; k < SY_K; ++k) {
      const int sw = k & 7;
      const float4 a0 = *(const float4*)(A + k * SY_B + 4 * (tr ^ sw)), a1 = *(const float4*)(A + k * SY_B + 4 * ((16 + tr) ^ sw));
      const float4 b0 = *(const float4*)(Bm + k * SY_B + 4 * (tc ^ sw)), b1 = *(const float4*)(Bm + k * SY_B + 4 * ((16 + tc) ^ sw));
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float bv[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 8; ++y) acc[8 * x + y] = fmaf(av[x], bv[y], acc[8 * x + y]);
      if (!diag)
#pragma unroll
        for (int x = 4; x < 8; ++x)
#pragma unroll
          for (int y = 0; y < 4; ++y) acc[8 * x + y] = fmaf(av[x], bv[y], acc[8 * x + y]);
#pragma unroll
      for (int x = 4; x < 8; ++x)
#pragma unroll
        for (int y = 4; y < 8; ++y) acc[8 * x + y] = fmaf(av[x], bv[y], acc[8 * x + y]);
    }
#pragma unroll
    for (int x = 0; x < 64; ++x) two_sum(hi[x], lo[x], acc[x]);
  }
  double* out = part + ((int64_t)blockIdx.x * ksplit + blockIdx.y) * SY_B * SY_B;
#pragma unroll
  for (int x = 0; x < 8; ++x)
#pragma unroll
    for (int y = 0; y < 8; ++y) {
      const int i = (x < 4 ? 4 * tr + x : 60 + 4 * tr + x), j = (y < 4 ? 4 * tc + y : 60 + 4 * tc + y);
      out[i + SY_B * j] = (double)hi[8 * x + y] + (double)lo[8 * x + y];
    }
}

// Sum the slices: C64, full n x n, from the entries on and above the diagonal.  32 entries a
// CTA, eight groups of slices side by side.
template <int T>                  // the tile size
__global__ void __launch_bounds__(256) k_syrk_finish(int64_t Nn, int ntile, int ksplit, const double* __restrict__ part,
                                                     double* __restrict__ C64) {
  __shared__ double sh[8][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int64_t e0 = blockIdx.x * (int64_t)32; e0 < Nn * Nn; e0 += gridDim.x * (int64_t)32) {
    const int64_t i = (e0 + lane) % Nn, j = (e0 + lane) / Nn;
    const bool in = j < Nn && i <= j;
    double s = 0.0;
    if (in) {
      const int ti = (int)(i / T), tj = (int)(j / T);
      const int pair = ti * ntile - ti * (ti - 1) / 2 + (tj - ti);
      const double* src = part + (int64_t)pair * ksplit * T * T + i % T + T * (j % T);
#pragma unroll 8
      for (int k = w; k < ksplit; k += 8) s += src[(int64_t)k * T * T];
    }
    __syncthreads();
    sh[w][lane] = s;
    __syncthreads();
    if (w == 0 && in) {
#pragma unroll
      for (int v = 1; v < 8; ++v) s += sh[v][lane];
      C64[i + Nn * j] = s;
      C64[j + Nn * i] = s;
    }
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
  const int64_t ncol = S / N[0];
  const int blocks = (int)std::min<int64_t>((ncol + 7) / 8, 152 * 8);
  const int vec = N[0] % 4 == 0 && ((uintptr_t)V & 15) == 0;      // (Vw and the weights are 256-byte aligned)
  k_weight_data<<<blocks, 256, 0, s>>>(V, sw, (unsigned)ncol, vec, Vw);
  count_launch();
}

// Tiles and column slices of a Gram: about one CTA per SM, a slice not below 128 columns.
struct GramSplit {
  int tile, ntile, npair, ksplit;
};
static GramSplit gram_shape(int64_t Nn, int64_t ncol) {
  GramSplit g;
  g.tile = Nn <= SY_T ? SY_T : SY_B;
  g.ntile = (int)((Nn + g.tile - 1) / g.tile);
  g.npair = g.ntile * (g.ntile + 1) / 2;
  // (slices rounded down where tiles of 128 fill the SMs once: a second, partial wave costs more)
  const int want = g.tile == SY_T ? (152 + g.npair - 1) / g.npair : std::max(1, 152 / g.npair);
  g.ksplit = (int)std::max<int64_t>(1, std::min<int64_t>(want, (ncol + 127) / 128));
  return g;
}

size_t gram_part_elems(int64_t Nn, int64_t ncol) {
  const GramSplit g = gram_shape(Nn, ncol);
  return (size_t)g.npair * g.ksplit * g.tile * g.tile;
}

void launch_gram_weighted(const float* Vw, int64_t L, int64_t Nn, int64_t Q, double* part, double* C64,
                          cudaStream_t s) {
  const GramSplit g = gram_shape(Nn, L * Q);
  const int blocks = (int)std::min<int64_t>((Nn * Nn + 31) / 32, 152 * 8);
  if (g.tile == SY_T) {
    k_syrk_partial<<<dim3(g.npair, g.ksplit), 256, 0, s>>>(Vw, L, Nn, Q, g.ntile, g.ksplit, part);
    count_launch();
    k_syrk_finish<SY_T><<<blocks, 256, 0, s>>>(Nn, g.ntile, g.ksplit, part, C64);
  } else {
    static bool attr = false;
    if (!attr) {
      cudaFuncSetAttribute(k_syrk_big, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSyrkBigSmem);
      attr = true;
    }
    k_syrk_big<<<dim3(g.npair, g.ksplit), 256, kSyrkBigSmem, s>>>(Vw, L, Nn, Q, g.ntile, g.ksplit, part);
    count_launch();
    k_syrk_finish<SY_B><<<blocks, 256, 0, s>>>(Nn, g.ntile, g.ksplit, part, C64);
  }
  count_launch();
}

}  // namespace tdb
