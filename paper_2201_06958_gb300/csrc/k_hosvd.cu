// k_hosvd.cu - truncated HOSVD used to initialise and re-initialise the bases
// (Sec. 2.3 last paragraph, Sec. 2.5), on the weighted mode-n Gram matrices
//     C_n = W_n^{1/2} V_(n) W_{-n} V_(n)^T W_n^{1/2}          (Sec. 2.6 names this matrix)
// whose eigenvalues are the squared mode-n singular values of the weighted data.
// The eigenproblems are in k_eig_modes.cu.
#include "common.cuh"
#include "kernels.h"

namespace tdb {

// ---------------------------------------------------------------------------
// Weighted mode-n Gram: partial 32x32 tiles over column slices, then finish.
// Column c of V_(n) is (l, q): V[l + L (i + N q)].
// ---------------------------------------------------------------------------

__device__ __forceinline__ double column_weight(const GramView& g, int64_t c) {
  int64_t l = c % g.L, q = c / g.L;
  double wc = 1.0;
  for (int m = 0; m < g.n; ++m) { wc *= g.w[m][l % g.N[m]]; l /= g.N[m]; }
  for (int m = g.n + 1; m < g.p; ++m) { wc *= g.w[m][q % g.N[m]]; q /= g.N[m]; }
  return wc;
}

// Bound: issue of the double multiply-adds (64 cycles a warp and sub-partition).  256 threads
// of 2 x 2 entries, so that four CTAs per SM cover each other's loads and barriers (1024
// threads of one entry left one CTA per SM: 126^3, one mode, 373 us, now 319); a diagonal tile forms the
// 528 entries on and above its diagonal only.
constexpr int WG_T = 256;
template <typename Tv>
__global__ void __launch_bounds__(WG_T, 4) k_wgram_partial(const Tv* __restrict__ V, const __grid_constant__ GramView g, int ntile, int ksplit,
                                                           double* __restrict__ part) {
  // blockIdx.x: upper tile pair (ti <= tj), blockIdx.y: column slice
  int t = blockIdx.x, ti = 0;
  while (t >= ntile - ti) { t -= ntile - ti; ++ti; }
  const int tj = ti + t;
  const bool diag = ti == tj;
  const int64_t i0 = (int64_t)ti * 32, j0 = (int64_t)tj * 32;
  const int64_t ncol = g.L * g.Q;
  const int64_t c0 = ncol * blockIdx.y / ksplit, c1 = ncol * (blockIdx.y + 1) / ksplit;
  __shared__ Tv As[32][33];
  __shared__ Tv Bs[32][33];
  __shared__ double wcol[32];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  // entries (bx | bx + 16, by | by + 16); on a diagonal tile (bx, by + 16), and of thread
  // t < 136 (ax, ay) and (ax + 16, ay + 16) with ax <= ay
  const int bx = threadIdx.x & 15, by = threadIdx.x >> 4;
  int ay = (int)((sqrtf(8.f * (float)threadIdx.x + 1.f) - 1.f) * 0.5f);
  while ((ay + 1) * (ay + 2) / 2 <= (int)threadIdx.x) ++ay;
  while (ay * (ay + 1) / 2 > (int)threadIdx.x) --ay;
  const int ax = (int)threadIdx.x - ay * (ay + 1) / 2;
  double acc00 = 0.0, acc01 = 0.0, acc10 = 0.0, acc11 = 0.0;
  const bool ifast = (g.L == 1);
  // columns fast: this thread's column is cb + tx, kept as (l, q)
  int64_t l = ifast ? 0 : (c0 + tx) % g.L, q = ifast ? 0 : (c0 + tx) / g.L;
  const int64_t dl = 32 % g.L, dq = 32 / g.L;
  for (int64_t cb = c0; cb < c1; cb += 32) {
    Tv va[4], vb[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int ri = ifast ? tx : ty + 8 * u;
      const int64_t c = cb + (ifast ? ty + 8 * u : tx);
      const int64_t ia = i0 + ri, ib = j0 + ri;
      const int64_t at = ifast ? g.Nn * c : l + g.L * g.Nn * q;
      va[u] = (c < c1 && ia < g.Nn) ? V[at + g.L * ia] : Tv(0);
      vb[u] = (c < c1 && ib < g.Nn) ? V[at + g.L * ib] : Tv(0);
    }
    l += dl;
    q += dq;
    if (l >= g.L) { l -= g.L; ++q; }
    if (threadIdx.x < 32) {
      const int64_t c = cb + threadIdx.x;
      wcol[threadIdx.x] = (c < c1) ? column_weight(g, c) : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int ri = ifast ? tx : ty + 8 * u, cc = ifast ? ty + 8 * u : tx;
      As[ri][cc] = (Tv)((double)va[u] * wcol[cc]);
      Bs[ri][cc] = vb[u];
    }
    __syncthreads();
    if (!diag) {
      Tv s00 = 0, s01 = 0, s10 = 0, s11 = 0;
#pragma unroll 8
      for (int k = 0; k < 32; ++k) {
        const Tv a0 = As[bx][k], a1 = As[bx + 16][k], b0 = Bs[by][k], b1 = Bs[by + 16][k];
        s00 += a0 * b0;
        s01 += a0 * b1;
        s10 += a1 * b0;
        s11 += a1 * b1;
      }
      acc00 += (double)s00;
      acc01 += (double)s01;
      acc10 += (double)s10;
      acc11 += (double)s11;
    } else {
      Tv s = 0;
#pragma unroll 8
      for (int k = 0; k < 32; ++k) s += As[bx][k] * Bs[by + 16][k];
      acc01 += (double)s;
      if (ay < 16) {
        Tv s00 = 0, s11 = 0;
#pragma unroll 8
        for (int k = 0; k < 32; ++k) {
          s00 += As[ax][k] * Bs[ay][k];
          s11 += As[ax + 16][k] * Bs[ay + 16][k];
        }
        acc00 += (double)s00;
        acc11 += (double)s11;
      }
    }
    __syncthreads();
  }
  double* out = part + ((int64_t)blockIdx.x * ksplit + blockIdx.y) * 1024;
  out[bx + 32 * (by + 16)] = acc01;
  if (!diag) {
    out[bx + 32 * by] = acc00;
    out[bx + 16 + 32 * by] = acc10;
    out[bx + 16 + 32 * (by + 16)] = acc11;
  } else if (ay < 16) {
    out[ax + 32 * ay] = acc00;
    out[ax + 16 + 32 * (ay + 16)] = acc11;
  }
}

// The slices' sums, scaled, for the entries on and above the diagonal, and mirrored: 32 entries
// a CTA, eight groups of slices side by side.
__global__ void __launch_bounds__(256) k_wgram_finish(GramView g, int ntile, int ksplit, const double* __restrict__ part,
                                                      double* __restrict__ C64) {
  __shared__ double sh[8][33];
  const int64_t Nn = g.Nn;
  const double* wn = g.w[g.n];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int64_t e0 = blockIdx.x * (int64_t)32; e0 < Nn * Nn; e0 += gridDim.x * (int64_t)32) {
    const int64_t i = (e0 + lane) % Nn, j = (e0 + lane) / Nn;
    const bool in = j < Nn && i <= j;
    double s = 0.0;
    if (in) {
      const int ti = (int)(i / 32), tj = (int)(j / 32);
      const int pair = ti * ntile - ti * (ti - 1) / 2 + (tj - ti);
      const double* src = part + (int64_t)pair * ksplit * 1024 + i % 32 + 32 * (j % 32);
#pragma unroll 8
      for (int k = w; k < ksplit; k += 8) s += src[(int64_t)k * 1024];
    }
    __syncthreads();
    sh[w][lane] = s;
    __syncthreads();
    if (w == 0 && in) {
#pragma unroll
      for (int v = 1; v < 8; ++v) s += sh[v][lane];
      s *= sqrt(wn[i] * wn[j]);
      C64[i + Nn * j] = s;
      C64[j + Nn * i] = s;
    }
  }
}

template <typename Tv>
void launch_wgram(const Tv* V, const GramView& g, double* part, size_t part_cap, double* C64, cudaStream_t s) {
  int ntile = (int)((g.Nn + 31) / 32);
  int npair = ntile * (ntile + 1) / 2;
  int64_t ncol = g.L * g.Q;
  int ksplit = (int)std::max<int64_t>(1, std::min<int64_t>((152 * 4 + npair - 1) / npair, (ncol + 255) / 256));
  while ((size_t)npair * ksplit * 1024 > part_cap && ksplit > 1) --ksplit;
  k_wgram_partial<Tv><<<dim3(npair, ksplit), WG_T, 0, s>>>(V, g, ntile, ksplit, part); count_launch();
  const int blocks = (int)std::min<int64_t>((g.Nn * g.Nn + 31) / 32, 152 * 8);
  k_wgram_finish<<<blocks, 256, 0, s>>>(g, ntile, ksplit, part, C64); count_launch();
}
template void launch_wgram<double>(const double*, const GramView&, double*, size_t, double*, cudaStream_t);

// U = W^{-1/2} Q[:, :r] (before the Cholesky-QR that makes U^T W U = I exact)
__global__ void k_scale_basis(const double* __restrict__ Q, const double* __restrict__ w, int64_t n, int r,
                              double* __restrict__ U) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n * r; e += (int64_t)gridDim.x * blockDim.x) {
    int64_t i = e % n;
    U[e] = Q[e] / sqrt(w[i]);
  }
}
void launch_scale_basis(const double* Q, const double* w, int64_t n, int r, double* U, cudaStream_t s) {
  int blocks = (int)std::min<int64_t>((n * r + 255) / 256, 1024);
  if (blocks < 1) blocks = 1;
  k_scale_basis<<<blocks, 256, 0, s>>>(Q, w, n, r, U); count_launch();
}

// ---------------------------------------------------------------------------
// A long first or last mode n (more points than the product M of the other modes) from
// the short side: with B = W_n^{1/2} V_(n) W_{-n}^{1/2} (N_n x M), C_n = B B^T has the
// nonzero eigenvalues of K = B^T B (M x M) and, for K z = lambda z, the unit eigenvector
// B z / sqrt(lambda) - the left singular vectors of B.  So the HOSVD of such a mode needs
// K, its leading eigenpairs and one product with B, never the N_n x N_n matrix.
// Column q of B^T is the merged index of the other modes, whose weight is
// w_q = prod_{m != n} w_m (i_m) with q = i_a + N_a (i_b + ...) over those modes in order.
// ---------------------------------------------------------------------------
__global__ void k_merge_weights(WeightView wv, int skip, int64_t M, double* __restrict__ wq) {
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < M; c += (int64_t)gridDim.x * blockDim.x) {
    int64_t idx = c;
    double w = 1.0;
    for (int m = 0; m < wv.p; ++m) {
      if (m == skip) continue;
      w *= wv.w[m][idx % wv.N[m]];
      idx /= wv.N[m];
    }
    wq[c] = w;
    wq[M + c] = sqrt(w);
  }
}
void launch_merge_weights(const WeightView& wv, int skip, int64_t M, double* wq, cudaStream_t s) {
  const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((M + 255) / 256, 1024));
  k_merge_weights<<<blocks, 256, 0, s>>>(wv, skip, M, wq); count_launch();
}

// Q[:, j] = B Z[:, j] / sqrt(lambda_j) in double.  Element (i, q) of B is
// V[i + N_n q] (first mode) or V[q + M i] (last mode), times sqrt(w_n(i) w_q) when the
// weights are given (sqw_q = sqrt(w_q)), else V is already weighted.
template <typename Tv>
__global__ void k_short_map(const Tv* __restrict__ V, int first, int64_t Nn, int64_t M, const double* __restrict__ wn,
                            const double* __restrict__ sqw, const double* __restrict__ Z, const double* __restrict__ ev,
                            int k, double* __restrict__ Q) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < Nn; i += (int64_t)gridDim.x * blockDim.x) {
    const double si = wn ? sqrt(wn[i]) : 1.0;
    for (int j = 0; j < k; ++j) {
      const double* z = Z + M * j;
      double acc = 0.0;
      for (int64_t q = 0; q < M; ++q) {
        const double v = (double)V[first ? i + Nn * q : q + M * i];
        acc = fma(sqw ? v * sqw[q] : v, z[q], acc);
      }
      const double lam = ev[j];
      Q[i + Nn * j] = lam > 0.0 ? si * acc / sqrt(lam) : 0.0;
    }
  }
}

// Each column scaled to unit length, its entry of largest magnitude made positive (the
// first such entry on ties), as for the eigenvectors of the direct route.
__global__ void k_col_unit_sign(double* __restrict__ Q, int64_t n) {
  __shared__ double red[32];
  __shared__ double bv[32];
  __shared__ long long bi[32];
  __shared__ long long imax;
  double* q = Q + n * blockIdx.x;
  double nrm = 0.0, best = -1.0;
  long long ib = 0x7fffffffffffffffll;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
    const double a = q[i];
    nrm += a * a;
    if (fabs(a) > best) { best = fabs(a); ib = i; }
  }
  nrm = block_sum(nrm, red);
  for (int o = 16; o > 0; o >>= 1) {
    const double ob = __shfl_xor_sync(0xffffffffu, best, o);
    const long long oi = __shfl_xor_sync(0xffffffffu, ib, o);
    if (ob > best || (ob == best && oi < ib)) { best = ob; ib = oi; }
  }
  if ((threadIdx.x & 31) == 0) { bv[threadIdx.x >> 5] = best; bi[threadIdx.x >> 5] = ib; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double b0 = bv[0];
    long long i0 = bi[0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
      if (bv[w] > b0 || (bv[w] == b0 && bi[w] < i0)) { b0 = bv[w]; i0 = bi[w]; }
    imax = i0 < n ? i0 : 0;      // (a column without a comparable entry has no largest one)
  }
  __syncthreads();
  const double sc = (q[imax] < 0.0 ? -1.0 : 1.0) / sqrt(nrm > 0.0 ? nrm : 1.0);
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) q[i] *= sc;
}

template <typename Tv>
void launch_short_map(const Tv* V, int first, int64_t Nn, int64_t M, const double* wn, const double* sqw,
                      const double* Z, const double* ev, int k, double* Q, cudaStream_t s) {
  const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((Nn + 127) / 128, 1024));
  k_short_map<Tv><<<blocks, 128, 0, s>>>(V, first, Nn, M, wn, sqw, Z, ev, k, Q); count_launch();
  k_col_unit_sign<<<k, 256, 0, s>>>(Q, Nn); count_launch();
}
template void launch_short_map<float>(const float*, int, int64_t, int64_t, const double*, const double*,
                                      const double*, const double*, int, double*, cudaStream_t);
template void launch_short_map<double>(const double*, int, int64_t, int64_t, const double*, const double*,
                                       const double*, const double*, int, double*, cudaStream_t);

}  // namespace tdb
