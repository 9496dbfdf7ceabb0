// k_eig_modes.cu - leading eigenpairs of the weighted mode Grams C_n (Secs. 2.3, 2.5) in
// double, every mode in one cooperative launch.
//
// Each mode has its own group of CTAs and group barrier; a CTA owns a few rows of the n x m
// block (m = k + 16 columns for k wanted pairs).  Per mode:
//   iterate  Z = C Q (every CTA its rows), Z^T Z and Q^T Z from the CTAs' partial sums, and
//            Q = orth(Z) by Cholesky-QR, repeated until the Gram it factored was close to the
//            identity (a first, ill-conditioned pass is shifted: the shifted CholeskyQR3 of
//            Fukaya, Kannan, Nakatsukasa, Yamamoto and Yanagisawa, SIAM J. Sci. Comput. 2020).
//            The iteration stops when the part of C q_j outside the block, relative to
//            C q_j, is below what the rounding of the Gram leaves of that eigenvector.
//   Ritz     H = Q^T C Q is diagonalised by a cyclic Jacobi on the group's first CTA, which
//            publishes its rotations sweep by sweep; the other CTAs apply them to their rows
//            of Q meanwhile, so no vector matrix is formed.
//   output   the k leading columns, unit length, entry of largest magnitude positive.
// A mode of at most m points skips the iteration (Q = I, H = C).  A mode of up to 96 points whose
// iteration has not settled after 30 rounds is solved whole in the same way: a spectrum that
// hardly decays (noise) would take hundreds, and its vectors were still off by up to 0.3 in angle.
// (A longer mode keeps the block that it has by then.)  In the float types pairs below 1e-5 of the
// largest eigenvalue are waited for three rounds at most once the others have settled: under a cap
// above the rank they are noise more often than not (float 1000 x 4 x 250 at rank 4, two pairs in
// noise: a re-initialisation 2.1 ms, waiting for them to the end 6.7 ms).
//
// Bound: chains of dependent double operations on one CTA (GB300 issues one double warp
// instruction per 64 cycles per SM sub-partition), so the design cuts the number of chains
// (iterations, factors, Jacobi sweeps) and runs the modes' chains side by side; the products
// are spread over all CTAs.  The result is a function of C alone, summed in a fixed order.
//
// Measured, all modes of a re-initialisation: 256 x 128 x 512 float (k = 18, 13, 10) 1.11 ms,
// where a float subspace iteration refined by double iterations and a one-CTA Jacobi, mode
// after mode in 130 launches, took 6.0 ms; 126^3 double (k = 7) 0.35 ms, where 24 iterations
// of single launches took 11.2 ms; 90^3 double against a one-CTA Jacobi of the whole Gram, a
// re-initialisation 1.1 against 76 ms.
#include "common.cuh"
#include "fastrcp.cuh"
#include "kernels.h"

namespace tdb {

namespace {

constexpr int EM_T = 256, EM_W = EM_T / 32;
constexpr int EM_M = kEigBlock;             // most columns of a block (50)
constexpr int EM_LD = EM_M + 1;             // leading dimension of m x m matrices in shared memory
constexpr int EM_RC = 8;                    // rows of C Z formed at a time
constexpr int EM_MP = (EM_M + 7) & ~7;      // columns padded to whole groups of eight (56)
constexpr int EM_ITERS = 30;                // iterations at most
constexpr int EM_SWEEPS = kEigSweeps;
constexpr double EM_TOL = 1e-15;            // off-diagonal mass left by the Jacobi
constexpr int EM_D = kEigWhole, EM_DLD = EM_D + 1;   // most points of a mode solved whole (96)

__device__ __forceinline__ unsigned em_ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void em_st_release(unsigned* p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void em_red_release(unsigned* p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Bounded wait of thread 0 until *word >= target; the outcome reaches every thread.
__device__ bool em_wait(const unsigned* word, unsigned target, unsigned* flags, volatile int* abort_sh) {
  if (threadIdx.x == 0) {
    const long long t0 = clock64();
    unsigned it = 0;
    while (em_ld_acquire(word) < target) {
      if ((++it & 31) == 0 && (clock64() - t0 > 4000000000ll || (em_ld_acquire(flags) & kFlagTimeout))) {
        atomicOr(flags, kFlagTimeout);
        *abort_sh = 1;
        break;
      }
    }
  }
  __syncthreads();
  return *abort_sh == 0;
}
// Group barrier: monotonic counter zeroed before the launch, the k-th waits for k * nct arrivals.
__device__ bool em_sync(unsigned* count, unsigned k, unsigned nct, unsigned* flags, volatile int* abort_sh) {
  __syncthreads();
  if (threadIdx.x == 0) em_red_release(count, 1u);
  return em_wait(count, k * nct, flags, abort_sh);
}

__device__ __forceinline__ double em_hash(uint32_t i, uint32_t j) {
  uint32_t h = i * 0x9E3779B1u ^ (j + 0x7F4A7C15u) * 0x85EBCA77u;
  h ^= h >> 15; h *= 0x2C1B3C6Du; h ^= h >> 12; h *= 0x297A2D39u; h ^= h >> 15;
  return (double)(h & 0xFFFFFF) / 8388608.0 - 1.0;   // [-1, 1)
}

// Order-preserving integer key of a double.
__device__ __forceinline__ long long em_key(double v) {
  const long long b = __double_as_longlong(v);
  return b >= 0 ? b : (long long)(b ^ 0x7fffffffffffffffLL);
}

// Zr (nr x m, ld mp) = C[r0 .. r0 + nr, :] Q.  Warp w takes an eighth of the n terms, its
// lanes eight columns x four terms; EM_RC rows in registers.  The four terms' sums are added
// by a transposing exchange (lane group kp ends with two of the eight rows), the warps'
// through shared memory (red: EM_W x EM_RC x mp), all in a fixed order.
__device__ void em_cz(const double* __restrict__ C, int n, const double* __restrict__ Q, int mp, int r0, int nr,
                      double* Zr, double* red) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int cl = lane & 7, kp = lane >> 3, NB = mp >> 3;
  const int l_lo = (int)((int64_t)n * w / EM_W), l_hi = (int)((int64_t)n * (w + 1) / EM_W);
  for (int rc = 0; rc < nr; rc += EM_RC) {
    const int nrc = min(EM_RC, nr - rc);
    double acc[EM_RC][EM_MP / 8];
#pragma unroll
    for (int x = 0; x < EM_RC; ++x)
#pragma unroll
      for (int b = 0; b < EM_MP / 8; ++b) acc[x][b] = 0.0;
    for (int l = l_lo + kp; l < l_hi; l += 4) {
      double q[EM_MP / 8];
#pragma unroll
      for (int b = 0; b < EM_MP / 8; ++b) q[b] = b < NB ? __ldcg(&Q[(int64_t)l * mp + 8 * b + cl]) : 0.0;
#pragma unroll
      for (int x = 0; x < EM_RC; ++x) {
        if (x >= nrc) break;
        const double c = __ldg(&C[(int64_t)(r0 + rc + x) * n + l]);     // (C is symmetric)
#pragma unroll
        for (int b = 0; b < EM_MP / 8; ++b)
          if (b < NB) acc[x][b] = fma(c, q[b], acc[x][b]);
      }
    }
    __syncwarp();
    const bool u16 = lane & 16, u8 = lane & 8;
#pragma unroll
    for (int b = 0; b < EM_MP / 8; ++b) {
      if (b >= NB) break;
      double h[4], g[2];
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const double keep = u16 ? acc[x + 4][b] : acc[x][b], send = u16 ? acc[x][b] : acc[x + 4][b];
        h[x] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
      }
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const double keep = u8 ? h[x + 2] : h[x], send = u8 ? h[x] : h[x + 2];
        g[x] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
      }
      const int row = (u16 ? 4 : 0) + (u8 ? 2 : 0);
      red[(w * EM_RC + row) * mp + 8 * b + cl] = g[0];
      red[(w * EM_RC + row + 1) * mp + 8 * b + cl] = g[1];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < nrc * mp; e += EM_T) {
      double s = red[e];
#pragma unroll
      for (int v = 1; v < EM_W; ++v) s += red[v * EM_RC * mp + e];
      Zr[rc * mp + e] = s;
    }
    __syncthreads();
  }
}

// part[e] = A^T B over this CTA's nr staged rows: the upper triangle (sym) or all of m x m.
// Entry (i, j) of the upper triangle is i + j (j + 1) / 2, of the full matrix i + m j.
__device__ void em_partial(const double* A, const double* B, int nr, int m, int mp, bool sym, double* part) {
  for (int e = threadIdx.x; e < m * m; e += EM_T) {
    const int i = e % m, j = e / m;
    if (sym && i > j) continue;
    double s = 0.0;
    for (int r = 0; r < nr; ++r) s = fma(A[r * mp + i], B[r * mp + j], s);
    part[sym ? i + j * (j + 1) / 2 : e] = s;
  }
}

// out[e] = sum over the group's CTAs of their partials (stride ps), for this CTA's share of
// the ne entries: a warp per entry, lanes over CTAs, then a butterfly (a fixed order).
__device__ void em_reduce(const double* part, int64_t ps, int nct, int cta, int ne, double* out) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int lo = (int)((int64_t)ne * cta / nct), hi = (int)((int64_t)ne * (cta + 1) / nct);
  for (int e = lo + w; e < hi; e += EM_W) {
    double s = 0.0;
    for (int c = lane; c < nct; c += 32) s += __ldcg(&part[ps * c + e]);
    s = warp_sum(s);
    if (lane == 0) out[e] = s;
  }
}

// X (upper triangular, X[i + EM_LD j]) with X^T G X = I from the symmetric G (full, ld EM_LD):
// Gaussian elimination of [D^-1 G D^-1 + shift I | I] without pivoting gives [U | E] with
// E = L^-1, X = D^-1 E^T U_d^-1/2.  Step k updates columns k + 1 .. k + m of the rows below
// (one multiply-add per entry; the multipliers are formed first, and the thread that updates
// the next pivot forms its reciprocal meanwhile).  A pivot that is not positive restarts with
// a larger shift; on the last attempt its column of X is zero.  R: m x 2m (ld EM_LD).
__device__ void em_factor(int m, const double* G, double shift0, double* R, double* X, double* dsc, double* mult,
                          unsigned* flags) {
  __shared__ double ip_sh[2];
  const int t = threadIdx.x;
  for (int i = t; i < m; i += EM_T) {
    const double g = G[i + EM_LD * i];
    dsc[i] = g > 0.0 ? drsqrt(g) : 1.0;
  }
  bool ok = false;
  for (int attempt = 0; attempt < 4 && !ok; ++attempt) {
    const double shift = attempt == 0 ? shift0 : (attempt == 1 ? fmax(1e-10, 100.0 * shift0) : (attempt == 2 ? 1e-5 : 1e-2));
    __syncthreads();
    for (int e = t; e < m * m; e += EM_T) {
      const int i = e % m, c = e / m;
      R[i + EM_LD * c] = G[i + EM_LD * c] * dsc[i] * dsc[c] + (i == c ? shift : 0.0);
      R[i + EM_LD * (m + c)] = i == c ? 1.0 : 0.0;
    }
    __syncthreads();
    if (t == 0) ip_sh[0] = drcp(R[0]);
    ok = true;
    for (int k = 0; k < m; ++k) {
      __syncthreads();
      const double piv = R[k + EM_LD * k];
      if (!(piv > 1e-300)) {
        ok = false;
        if (attempt < 3) break;
        if (t == 0 && k + 1 < m) ip_sh[(k + 1) & 1] = drcp(R[k + 1 + EM_LD * (k + 1)]);
        continue;
      }
      const int cnt = m - 1 - k;
      if (cnt == 0) break;
      if (t < cnt) mult[t] = R[k + 1 + t + EM_LD * k] * ip_sh[k & 1];
      __syncthreads();
      for (int e = t; e < cnt * m; e += EM_T) {
        const int ri = e % cnt, i = k + 1 + ri, c = k + 1 + e / cnt;
        const double v = fma(-mult[ri], R[k + EM_LD * c], R[i + EM_LD * c]);
        R[i + EM_LD * c] = v;
        if (e == 0) ip_sh[(k + 1) & 1] = drcp(v);
      }
    }
    __syncthreads();
  }
  if (!ok && t == 0) atomicOr(flags, kFlagEigNoConv);
  for (int j = t; j < m; j += EM_T) {
    const double u = R[j + EM_LD * j];
    mult[j] = u > 1e-300 ? drsqrt(u) : 0.0;
  }
  __syncthreads();
  for (int e = t; e < m * m; e += EM_T) {
    const int i = e % m, j = e / m;
    X[i + EM_LD * j] = j >= i ? dsc[i] * R[j + EM_LD * (m + i)] * mult[j] : 0.0;
  }
  __syncthreads();
}

// Pair k of round rd of the round-robin over nn (even) indices (Brent and Luk's ordering).
__device__ __forceinline__ void em_pair(int nn, int rd, int k, int& p, int& q) {
  if (k == 0) {
    p = rd;
    q = nn - 1;
  } else {
    p = rd + k;
    if (p >= nn - 1) p -= nn - 1;
    q = rd - k;
    if (q < 0) q += nn - 1;
  }
}

// (c, s) pairs of one sweep over m indices.
__host__ __device__ inline int64_t em_sweep_pairs(int m) {
  const int64_t nn = (m + 1) & ~1;
  return (nn - 1) * (nn / 2);
}

// One sweep's rotations (rounds x pairs of (c, s)) applied to the rows A (nr x m, ld mp): a
// warp per row, a lane per pair (or two).
__device__ void em_apply_sweep(double* A, int nr, int m, int mp, const double2* rot) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nn = (m + 1) & ~1, half = nn / 2;
  for (int r = w; r < nr; r += EM_W) {
    double* row = A + r * mp;
    for (int rd = 0; rd < nn - 1; ++rd) {
      for (int k = lane; k < half; k += 32) {
        int p, q;
        em_pair(nn, rd, k, p, q);
        const double2 cs = __ldcg(&rot[rd * half + k]);
        const double vp = row[p], vq = row[q];
        row[p] = fma(cs.x, vp, -(cs.y * vq));
        row[q] = fma(cs.y, vp, cs.x * vq);
      }
      __syncwarp();
    }
  }
}

// Cyclic Jacobi on the symmetric H (m x m, full, ld LDH; row and column nn - 1 zero for odd
// m; NB blocks of 2 x 2 a thread at most) by this CTA, the rotations of sweep s written to rot[s]
// and announced through *done (s + 1; the last one with kEmLast set).  Every pair rotates: the block's columns are not
// sorted, so a wanted Ritz value can sit in its tail.  The angle's tangent is a
// float root of b t^2 + (a_qq - a_pp) t - b = 0 with one Newton step in double, its cosine and
// sine are double.  The 2 x 2 blocks above the diagonal are updated and mirrored.  Ends when the
// off-diagonal mass is below tol^2 of the diagonal's, or at the rounding floor (below (m u)^2 of it
// and a sweep that does not quarter it).  A sweep higher up may well leave more than a quarter:
// graded or clustered spectra take up to 21 sweeps of 96 points, and ending them there (from the
// third sweep on) left one HOSVD in a hundred with subspaces off by up to 0.2.
constexpr unsigned kEmLast = 0x80000000u;
template <int NB, int LDH>
__device__ bool em_jacobi(double* H, int m, double tol, double2* rot, unsigned* done, double* cs, int* pq,
                          double* red) {
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int nn = (m + 1) & ~1, half = nn / 2, nblk = half * (half + 1) / 2;
  // this thread's blocks (I <= J), the same in every round
  int blk[NB];
#pragma unroll
  for (int u = 0; u < NB; ++u) {
    const int e = t + EM_T * u;
    int J = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
    while ((J + 1) * (J + 2) / 2 <= e) ++J;
    while (J * (J + 1) / 2 > e) --J;
    blk[u] = e < nblk ? ((e - J * (J + 1) / 2) | (J << 8)) : -1;
  }
  const double floor2 = (1.2e-16 * m) * (1.2e-16 * m);
  double off_prev = 0.0;
  bool conv = false;
  for (int sweep = 0;; ++sweep) {
    double off = 0.0, dia = 0.0;
    for (int e = t; e < m * m; e += EM_T) {
      const int i = e % m, j = e / m;
      const double v = H[i + LDH * j];
      if (i == j) dia = fma(v, v, dia);
      else if (i < j) off = fma(v, v, off);
    }
    off = 2.0 * warp_sum(off);
    dia = warp_sum(dia);
    if (lane == 0) { red[w] = off; red[EM_W + w] = dia; }
    __syncthreads();
    off = 0.0;
    dia = 0.0;
#pragma unroll
    for (int v = 0; v < EM_W; ++v) { off += red[v]; dia += red[EM_W + v]; }
    conv = off <= tol * tol * dia || dia == 0.0;
    const bool stop = conv || sweep == EM_SWEEPS || (off <= floor2 * dia && off > 0.25 * off_prev);
    off_prev = off;
    __syncthreads();
    if (stop) {
      if (t == 0) em_st_release(done, (unsigned)sweep | kEmLast);
      return conv || sweep < EM_SWEEPS;
    }
    double2* out = rot + sweep * em_sweep_pairs(m);
    for (int rd = 0; rd < nn - 1; ++rd) {
      if (t < half) {
        int p, q;
        em_pair(nn, rd, t, p, q);
        const double app = H[p + LDH * p], aqq = H[q + LDH * q], apq = H[p + LDH * q];
        double c = 1.0, s = 0.0;
        const float fpq = (float)apq;
        if (fabsf(fpq) > 1e-30f && fpq * fpq > 1e-32f * fabsf((float)app * (float)aqq)) {
          const float theta = (float)(aqq - app) / (2.f * fpq);
          const float at = fabsf(theta);
          const float root = at < 1e18f ? sqrtf(fmaf(at, at, 1.f)) : at;
          const float t0 = copysignf(1.f / (at + root), theta);
          const double diff = aqq - app;
          const float slope = fmaf(2.f * fpq, t0, (float)diff);          // (both terms of t0's sign)
          const double tt = fma(-fma(fma(apq, (double)t0, diff), (double)t0, -apq), (double)(1.f / slope), (double)t0);
          c = drsqrt(fma(tt, tt, 1.0));
          s = tt * c;
        }
        cs[2 * t] = c;
        cs[2 * t + 1] = s;
        pq[2 * t] = p;
        pq[2 * t + 1] = q;
        out[rd * half + t] = make_double2(c, s);
      }
      __syncthreads();
#pragma unroll
      for (int u = 0; u < NB; ++u) {
        if (blk[u] < 0) continue;
        const int I = blk[u] & 255, J = blk[u] >> 8;
        const int pI = pq[2 * I], qI = pq[2 * I + 1], pJ = pq[2 * J], qJ = pq[2 * J + 1];
        const double cI = cs[2 * I], sI = cs[2 * I + 1], cJ = cs[2 * J], sJ = cs[2 * J + 1];
        const double b00 = H[pI + LDH * pJ], b01 = H[pI + LDH * qJ], b10 = H[qI + LDH * pJ],
                     b11 = H[qI + LDH * qJ];
        const double c00 = fma(cJ, b00, -(sJ * b01)), c01 = fma(sJ, b00, cJ * b01);
        const double c10 = fma(cJ, b10, -(sJ * b11)), c11 = fma(sJ, b10, cJ * b11);
        const double d00 = fma(cI, c00, -(sI * c10)), d01 = fma(cI, c01, -(sI * c11));
        const double d10 = fma(sI, c00, cI * c10), d11 = fma(sI, c01, cI * c11);
        H[pI + LDH * pJ] = d00;
        H[qI + LDH * qJ] = d11;
        H[pI + LDH * qJ] = d01;
        if (I == J) {
          H[qI + LDH * pI] = d01;
        } else {
          H[qI + LDH * pJ] = d10;
          H[pJ + LDH * pI] = d00;
          H[qJ + LDH * pI] = d01;
          H[pJ + LDH * qI] = d10;
          H[qJ + LDH * qI] = d11;
        }
      }
      __syncthreads();
    }
    if (t == 0) {
      __threadfence();
      em_st_release(done, (unsigned)(sweep + 1));
    }
  }
}

// Shared memory (doubles): the factor's [G | I], G, X, H (where C itself goes for a mode that is
// solved whole); the CTA's rows of Q and Z; the C Z reduction (all three the rows of the whole
// solve, if it comes to that).
__host__ __device__ constexpr size_t em_fixed() { return 5 * (size_t)EM_LD * EM_M + 64 + 64 + EM_D + 64; }
static_assert(5 * EM_LD * EM_M >= EM_DLD * EM_D, "C of a mode solved whole");
__host__ __device__ inline size_t em_smem(int n, int mp, int rows) {
  size_t v = 2 * (size_t)rows * mp + (size_t)EM_W * EM_RC * mp;
  const size_t whole = n <= EM_D ? (size_t)rows * ((n + 7) & ~7) : 0;
  if (v < whole) v = whole;
  return sizeof(double) * (em_fixed() + v);
}

__global__ void __launch_bounds__(EM_T, 1) k_eig_modes(EigModes a) {
  extern __shared__ __align__(16) double em_sm[];
  __shared__ int abort_sh, ord[EM_D], pq[128];
  __shared__ unsigned done_sh;
  int md = 0;
  while (md + 1 < a.p && (int)blockIdx.x >= a.mode[md + 1].cta0) ++md;
  const EigMode M = a.mode[md];
  const int B = M.nct, b = (int)blockIdx.x - M.cta0, n = M.n, m = M.m, k = M.k, mp = M.mp;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  double* R = em_sm;                         // m x 2m
  double* G = R + 2 * EM_LD * EM_M;          // Z^T Z
  double* X = G + EM_LD * EM_M;
  double* H = X + EM_LD * EM_M;              // Q^T Z
  double* dsc = H + EM_LD * EM_M;            // 64
  double* mult = dsc + 64;                   // 64
  double* cs = mult + 64;                    // EM_D (pairs' c, s)
  double* red = cs + EM_D;                   // 64 for sums
  double* Qr = red + 64;                     // this CTA's rows of Q (nr x mp)
  // the group's first CTA runs the Jacobi and owns no rows (a group has at least two)
  const int nb = B - 1;
  const int r_lo = b == 0 ? 0 : (int)((int64_t)n * (b - 1) / nb), r_hi = b == 0 ? 0 : (int)((int64_t)n * b / nb);
  const int nr = r_hi - r_lo;
  const int rows = (n + nb - 1) / nb;
  double* Zr = Qr + (size_t)rows * mp;
  double* czr = Zr + (size_t)rows * mp;
  if (t == 0) abort_sh = 0;
  __syncthreads();
  unsigned nbar = 0;
  const int ntri = m * (m + 1) / 2, nful = m * m;
  double* part = M.part + (int64_t)b * M.pstride;
  // A^T B of the staged rows summed over the group into G (upper, mirrored) and H (all)
  auto gather = [&](bool with_h) -> bool {
    em_partial(Zr, Zr, nr, m, mp, true, part);
    if (with_h) em_partial(Qr, Zr, nr, m, mp, false, part + ntri);
    if (!em_sync(M.bar, ++nbar, B, a.flags, &abort_sh)) return false;
    em_reduce(M.part, M.pstride, B, b, ntri + (with_h ? nful : 0), M.sums);
    if (!em_sync(M.bar, ++nbar, B, a.flags, &abort_sh)) return false;
    for (int e = t; e < nful; e += EM_T) {
      const int i = e % m, j = e / m;
      G[i + EM_LD * j] = __ldcg(&M.sums[i <= j ? i + j * (j + 1) / 2 : j + i * (i + 1) / 2]);
      if (with_h) H[i + EM_LD * j] = __ldcg(&M.sums[ntri + e]);
    }
    __syncthreads();
    return true;
  };
  double delta = 0.0;                        // the shift of the iterated matrix, below
  bool whole = m == n;                       // every vector is kept: Q = I, H = C
  if (!whole) {
    const double u = 1.1102230246251565e-16;
    const double s0 = 11.0 * ((double)n * m + (double)m * (m + 1)) * u * m;
    // C + delta I is iterated, delta one rounding of C's largest diagonal entry (the Ritz values
    // give it back): data that mirror exactly (32 points of an even function in float: rank 16
    // under a block of 24) leave C Q exactly deficient, which no Cholesky-QR repairs, and every
    // iteration ran all its passes: that re-initialisation 7.3 ms, with the shift 0.62 ms.
    for (int i = t; i < n; i += EM_T) delta = fmax(delta, fabs(__ldg(&M.C[i + (int64_t)n * i])));
    for (int o = 16; o > 0; o >>= 1) delta = fmax(delta, __shfl_xor_sync(0xffffffffu, delta, o));
    if (lane == 0) red[w] = delta;
    __syncthreads();
    for (int v = 0; v < EM_W; ++v) delta = fmax(delta, red[v]);
    delta *= 2.0 * u;
    __syncthreads();
    for (int e = t; e < nr * mp; e += EM_T) {
      const int row = r_lo + e / mp, c = e % mp;
      const double v = c < m ? em_hash((uint32_t)row, (uint32_t)c) : 0.0;
      Qr[e] = v;
      M.Q[(int64_t)row * mp + c] = v;
    }
    int extra = -1;                          // iterations still to do once the block has settled
    int waited = 0;                          // iterations since the columns above M.least have
    if (!em_sync(M.bar, ++nbar, B, a.flags, &abort_sh)) return;
    for (int it = 0;; ++it) {
      em_cz(M.C, n, M.Q, mp, r_lo, nr, Zr, czr);
      for (int e = t; e < nr * mp; e += EM_T) Zr[e] = fma(delta, Qr[e], Zr[e]);
      __syncthreads();
      if (!gather(it > 0)) return;
      if (it > 0) {
        // Settled: for every wanted column above the Gram's rounding, the part of z_j = C q_j
        // outside the block is below 2e-7 of it (what z_j^T z_j - |Q^T z_j|^2 can resolve is
        // a few 1e-8).  One iteration shrinks that part by lambda_out / lambda_j, lambda_out at most
        // the block's smallest Ritz value; as many follow as bring it below
        // tau lambda_1 / lambda_j, the perturbation of that eigenvector by the Gram's rounding.
        if (extra < 0) {
          double need = 0.0;
          bool settled = true, large = true;     // every wanted column, those above M.least
          double top = 0.0, low = H[0];
          for (int j = 0; j < m; ++j) {
            const double h = fmax(H[j + EM_LD * j], 0.0);
            top = fmax(top, h);
            low = fmin(low, h);
          }
          if (t < k) {
            const double hj = H[t + EM_LD * t];
            if (hj > 10.0 * M.tau * top) {
              double in = 0.0;
              for (int i = 0; i < m; ++i) in = fma(H[i + EM_LD * t], H[i + EM_LD * t], in);
              const double g = G[t + EM_LD * t];
              settled = g - in <= 4e-14 * g;
              large = settled || hj <= M.least * top;
              const float aim = (float)(M.tau * 5e6 * top / hj);      // relative to the 2e-7 reached
              if (aim < 1.f) {
                const float rate = fminf((float)(low / hj), 0.999f);
                need = rate < 1e-30f ? 1.0 : ceil(logf(aim) / logf(rate));
              }
            }
          }
          settled = __syncthreads_and(settled);
          large = __syncthreads_and(large);
          if (!settled && large && ++waited > 3) {
            extra = 0;
          } else if (settled) {
            // the largest count any column asks for
            if (t < 64) red[t] = t < k ? need : 0.0;
            __syncthreads();
            double worst = 0.0;
            for (int j = 0; j < k; ++j) worst = fmax(worst, red[j]);
            extra = (int)fmin(worst, (double)EM_ITERS);
            __syncthreads();
          }
        } else {
          --extra;
        }
        if (extra == 0) break;
        if (it == EM_ITERS) {
          whole = n <= EM_D;
          break;
        }
      }
      // Q = orth(Z)
      for (int pass = 0; pass < 6; ++pass) {
        double offd = 0.0;
        for (int e = t; e < nful; e += EM_T) {
          const int i = e % m, j = e / m;
          if (i < j) {
            const double g = G[i + EM_LD * j], d = G[i + EM_LD * i] * G[j + EM_LD * j];
            const float f = d > 0.0 ? (float)(g * g) / (float)d : 0.f;
            offd += (double)f;
          }
        }
        offd = warp_sum(offd);
        if (lane == 0) red[w] = offd;
        __syncthreads();
        offd = 0.0;
        for (int v = 0; v < EM_W; ++v) offd += red[v];
        const bool near = offd <= 0.0625;        // |D^-1 G D^-1 - I|_F <= 0.36: one factor suffices
        __syncthreads();
        em_factor(m, G, near ? 0.0 : (pass == 0 ? s0 : 0.0), R, X, dsc, mult, a.flags);
        for (int e = t; e < nr * mp; e += EM_T) {
          const int r = e / mp, c = e % mp;
          double s = 0.0;
          if (c < m)
            for (int l = 0; l <= c; ++l) s = fma(Zr[r * mp + l], X[l + EM_LD * c], s);
          Qr[e] = s;
        }
        __syncthreads();
        if (near || pass == 5) break;
        for (int e = t; e < nr * mp; e += EM_T) Zr[e] = Qr[e];
        __syncthreads();
        if (!gather(false)) return;
      }
      for (int e = t; e < nr * mp; e += EM_T) M.Q[(int64_t)(r_lo + e / mp) * mp + e % mp] = Qr[e];
      if (!em_sync(M.bar, ++nbar, B, a.flags, &abort_sh)) return;
    }
    if (!whole) {
      for (int e = t; e < nful; e += EM_T) {
        const int i = e % m, j = e / m;
        if (i < j) {
          const double h = 0.5 * (H[i + EM_LD * j] + H[j + EM_LD * i]);
          H[i + EM_LD * j] = h;
          H[j + EM_LD * i] = h;
        }
      }
      __syncthreads();
    }
  }
  // the matrix to diagonalise: dm x dm at Hd (ld dld), the rows of its basis at Qr (ld dmp)
  int dm = m, dmp = mp, dld = EM_LD;
  double* Hd = H;
  if (whole) {
    dm = n;
    dmp = (n + 7) & ~7;
    if (n > EM_M) {
      dld = EM_DLD;
      Hd = em_sm;
    }
    delta = 0.0;
    __syncthreads();
    for (int e = t; e < nr * dmp; e += EM_T) Qr[e] = (r_lo + e / dmp == e % dmp) ? 1.0 : 0.0;
    if (b == 0)
      for (int e = t; e < n * n; e += EM_T) Hd[(e % n) + dld * (e / n)] = M.C[e];
    __syncthreads();
  }
  // Ritz values and vectors
  double2* rot = (double2*)M.rot;
  int* order = (int*)(M.sums + kEigPart - 64);        // past the sums
  auto apply_from = [&](unsigned have, unsigned upto) {
    for (unsigned s = have; s < upto; ++s)
      em_apply_sweep(Qr, nr, dm, dmp, rot + s * em_sweep_pairs(dm));
  };
  if (b == 0) {
    // scaled by a power of two so that the float angles neither overflow nor vanish
    int ex = 0;
    {
      double big = 0.0;
      for (int j = 0; j < dm; ++j) big = fmax(big, fabs(Hd[j + dld * j]));
      if (big > 0.0 && isfinite(big)) frexp(big, &ex);
    }
    __syncthreads();
    const double sc = ldexp(1.0, -ex), un = ldexp(1.0, ex);
    const int nn = (dm + 1) & ~1;
    for (int e = t; e < nn * nn; e += EM_T) {
      const int i = e % nn, j = e / nn;
      Hd[i + dld * j] = (i < dm && j < dm) ? Hd[i + dld * j] * sc : 0.0;
    }
    __syncthreads();
    const bool conv = dm > EM_M ? em_jacobi<5, EM_DLD>(Hd, dm, EM_TOL, rot, M.done, cs, pq, red)
                                : em_jacobi<2, EM_LD>(Hd, dm, EM_TOL, rot, M.done, cs, pq, red);
    if (!conv && t == 0) atomicOr(a.flags, kFlagEigNoConv);
    // descending order by integer keys, ties by index: a permutation whatever the values
    for (int j = t; j < dm; j += EM_T) {
      const long long kj = em_key(Hd[j + dld * j]);
      int rank = 0;
      for (int l = 0; l < dm; ++l) {
        const long long kl = em_key(Hd[l + dld * l]);
        rank += (kl > kj) || (kl == kj && l < j);
      }
      order[rank] = j;
      if (rank < k) M.ev[rank] = Hd[j + dld * j] * un - delta;
    }
  } else {
    unsigned have = 0;
    for (;;) {
      if (!em_wait(M.done, have + 1, a.flags, &abort_sh)) return;
      if (t == 0) done_sh = em_ld_acquire(M.done);
      __syncthreads();
      const unsigned d = done_sh;
      __syncthreads();
      apply_from(have, d & ~kEmLast);
      have = d & ~kEmLast;
      if (d & kEmLast) break;
    }
  }
  // trace of C
  if (b == B - 1 && w == 0) {
    double s = 0.0;
    for (int i = lane; i < n; i += 32) s += M.C[i + (int64_t)n * i];
    s = warp_sum(s);
    if (lane == 0) *M.trace = s;
  }
  if (!em_sync(M.bar, ++nbar, B, a.flags, &abort_sh)) return;
  for (int j = t; j < dm; j += EM_T) ord[j] = __ldcg(&order[j]);
  __syncthreads();
  // per-CTA column sums of squares, largest |entry| and its row
  double* col = M.part + (int64_t)b * M.pstride;
  for (int j = t; j < k; j += EM_T) {
    double nrm = 0.0, best = -1.0;
    int ib = 0x7fffffff;
    for (int r = 0; r < nr; ++r) {
      const double v = Qr[r * dmp + ord[j]];
      nrm = fma(v, v, nrm);
      if (fabs(v) > best) { best = fabs(v); ib = r_lo + r; }
    }
    col[j] = nrm;
    col[EM_M + j] = best;
    col[2 * EM_M + j] = ib < n ? (double)ib : (double)n;
    col[3 * EM_M + j] = ib < n && Qr[(ib - r_lo) * dmp + ord[j]] < 0.0 ? -1.0 : 1.0;
  }
  if (!em_sync(M.bar, ++nbar, B, a.flags, &abort_sh)) return;
  for (int j = w; j < k; j += EM_W) {
    double nrm = 0.0, best = -2.0, sg = 1.0;
    int ib = 0x7fffffff;
    for (int c = lane; c < B; c += 32) {
      const double* o = M.part + (int64_t)c * M.pstride;
      nrm += __ldcg(&o[j]);
      const double v = __ldcg(&o[EM_M + j]);
      const int i = (int)__ldcg(&o[2 * EM_M + j]);
      if (v > best || (v == best && i < ib)) { best = v; ib = i; sg = __ldcg(&o[3 * EM_M + j]); }
    }
    nrm = warp_sum(nrm);
    for (int o = 16; o > 0; o >>= 1) {
      const double ob = __shfl_xor_sync(0xffffffffu, best, o), os = __shfl_xor_sync(0xffffffffu, sg, o);
      const int oi = __shfl_xor_sync(0xffffffffu, ib, o);
      if (ob > best || (ob == best && oi < ib)) { best = ob; ib = oi; sg = os; }
    }
    if (lane == 0) dsc[j] = sg / sqrt(nrm > 0.0 ? nrm : 1.0);
  }
  __syncthreads();
  for (int e = t; e < nr * k; e += EM_T) {
    const int r = e % nr, j = e / nr;
    M.out[r_lo + r + (int64_t)n * j] = Qr[r * dmp + ord[j]] * dsc[j];
  }
}

int em_cols(int n, int k) { return std::min(n, k + 16); }

// The CTAs of each mode (the Jacobi's and those that own rows), and the shared memory of the
// launch.  A row CTA holds its rows of Q and Z in shared memory, so a mode takes at least the CTAs
// that its rows need for that (110 rows and more of the widest block fill one); past that the SMs
// are shared in proportion to n^2, the entries of C that a product reads, and a mode whose vectors
// are all kept (no products) takes no more than leave eight rows, one per warp, to a CTA.  (By n^2
// alone a mode of 119 points beside one of 1024 got one CTA, and the launch was refused.)
// False: not on this many SMs.
struct EmSplit {
  int nct[kMaxModes];
  size_t smem;
};
bool em_split(const int* n, const int* k, int p, int nsm, size_t limit, EmSplit& out) {
  double tot = 0.0;
  for (int i = 0; i < p; ++i) tot += (double)n[i] * n[i];
  const int avail = nsm - 2 * p;
  int need[kMaxModes], sum = 0;
  for (int i = 0; i < p; ++i) {
    const int m = em_cols(n[i], k[i]), mp = (m + 7) & ~7;
    int rows = n[i];                         // the most rows of a CTA
    while (rows > 0 && em_smem(n[i], mp, rows) > limit) --rows;
    if (rows == 0) return false;
    need[i] = (n[i] + rows - 1) / rows;
    const int want = avail > 0 ? (int)((double)avail * ((double)n[i] * n[i] / tot)) : 0;
    const int most = m == n[i] ? (n[i] + EM_W - 1) / EM_W : n[i];
    out.nct[i] = 1 + std::max(need[i], std::min(std::max(want, 1), most));
    sum += out.nct[i];
  }
  for (; sum > nsm; --sum) {                 // the mode with the most to spare gives one up
    int best = 0;
    for (int i = 1; i < p; ++i)
      if (out.nct[i] - need[i] > out.nct[best] - need[best]) best = i;
    if (out.nct[best] - 1 <= need[best]) return false;
    --out.nct[best];
  }
  out.smem = 0;
  for (int i = 0; i < p; ++i) {
    const int nb = out.nct[i] - 1, mp = (em_cols(n[i], k[i]) + 7) & ~7;
    out.smem = std::max(out.smem, em_smem(n[i], mp, (n[i] + nb - 1) / nb));
  }
  return true;
}

}  // namespace

// A CTA's partial sums: the block's m x m and its upper triangle, or four statistics a column.
// (Even: the rotations that follow are read 16 bytes at a time.)
static int em_pstride(int m) { return (std::max(m * (m + 1) / 2 + m * m, 4 * EM_M) + 1) & ~1; }
static_assert(EM_M * (EM_M + 1) / 2 + EM_M * EM_M + 64 <= kEigPart && EM_D <= 128, "the sums, and the order after them");

size_t eig_modes_scratch(int n, int k) {
  const size_t m = em_cols(n, k), mp = (m + 7) & ~(size_t)7;
  return (size_t)n * mp + (size_t)std::min(152, n + 1) * em_pstride((int)m) + kEigPart +
         (size_t)kEigSweeps * 2 * em_sweep_pairs(n <= EM_D ? n : (int)m) + 8;
}

tdb_status launch_eig_modes(EigProblem* pr, int p, double tau, double least, unsigned* flags, cudaStream_t s) {
  // (read once; what the device gives less than 2 KB for the kernel's static shared memory)
  struct Device {
    int nsm = 0, coop = 0;
    size_t optin = 0;
  };
  static const Device dev = [] {
    Device d;
    int id = 0, lim = 0;
    cudaGetDevice(&id);
    cudaDeviceGetAttribute(&d.nsm, cudaDevAttrMultiProcessorCount, id);
    cudaDeviceGetAttribute(&d.coop, cudaDevAttrCooperativeLaunch, id);
    cudaDeviceGetAttribute(&lim, cudaDevAttrMaxSharedMemoryPerBlockOptin, id);
    d.nsm = std::min(d.nsm, 152);
    d.optin = (size_t)std::max(lim - 2048, 0);
    return d;
  }();
  if (!dev.coop) return TDB_ERR_UNSUPPORTED;
  int n[kMaxModes], k[kMaxModes];
  for (int i = 0; i < p; ++i) {
    n[i] = pr[i].n;
    k[i] = pr[i].k;
    if (k[i] > n[i] || em_cols(n[i], k[i]) > EM_M) return TDB_ERR_INVALID_ARG;
  }
  EmSplit split;
  if (!em_split(n, k, p, dev.nsm, dev.optin, split)) return TDB_ERR_UNSUPPORTED;
  EigModes a;
  a.p = p;
  a.flags = flags;
  int cta = 0;
  for (int i = 0; i < p; ++i) {
    EigMode& M = a.mode[i];
    M.C = pr[i].C;
    M.n = pr[i].n;
    M.k = pr[i].k;
    M.m = em_cols(M.n, M.k);
    M.mp = (M.m + 7) & ~7;
    M.nct = split.nct[i];
    M.cta0 = cta;
    cta += M.nct;
    double* w = pr[i].scratch;
    M.Q = w;
    w += (size_t)M.n * M.mp;
    M.part = w;
    M.pstride = em_pstride(M.m);
    w += (size_t)std::min(152, M.n + 1) * M.pstride;
    M.sums = w;
    w += kEigPart;
    M.rot = w;
    w += (size_t)kEigSweeps * 2 * em_sweep_pairs(M.n <= EM_D ? M.n : M.m);
    M.bar = (unsigned*)w;
    M.done = M.bar + 4;
    M.ev = pr[i].ev;
    M.out = pr[i].Q;
    M.trace = pr[i].trace;
    M.tau = tau;
    M.least = least;
    cudaMemsetAsync(M.bar, 0, 8 * sizeof(unsigned), s);
  }
  // (the limit, not this launch's need: another thread's launch may need more)
  cudaFuncSetAttribute(k_eig_modes, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dev.optin);
  void* args[] = {(void*)&a};
  const cudaError_t e = cudaLaunchCooperativeKernel((const void*)k_eig_modes, cta, EM_T, args, split.smem, s);
  count_launch();
  return e == cudaSuccess ? TDB_OK : TDB_ERR_CUDA;
}

}  // namespace tdb

extern "C" tdb_status tdb_selftest_eig_split(int nmodes, const int* n, const int* k, int num_sms,
                                             int64_t smem_bytes, int* ctas, int64_t* smem) {
  using namespace tdb;
  if (nmodes < 1 || nmodes > kMaxModes || !n || !k || !ctas || !smem || num_sms < 1 || smem_bytes < 1)
    return TDB_ERR_INVALID_ARG;
  for (int i = 0; i < nmodes; ++i)
    if (n[i] < 1 || k[i] < 1 || k[i] > n[i] || em_cols(n[i], k[i]) > EM_M) return TDB_ERR_INVALID_ARG;
  EmSplit split;
  if (!em_split(n, k, nmodes, num_sms, (size_t)smem_bytes, split)) return TDB_ERR_UNSUPPORTED;
  for (int i = 0; i < nmodes; ++i) ctas[i] = split.nct[i];
  *smem = (int64_t)split.smem;
  return TDB_OK;
}
