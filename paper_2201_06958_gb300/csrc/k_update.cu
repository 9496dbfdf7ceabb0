// k_update.cu - the rank-sized algebra of one step in one cooperative launch.
//
// Rows of every mode are split in tiles of 32 over all CTAs, r x r work runs on
// one CTA per mode, and bounded grid barriers separate the phases.  Tc is the
// compute type (float or double); the state (U, T, R, R^{-1}, G^{-1}) is double.
//   1 rows : M = Y_(n) T_(n)^T, X = M G_n^{-1}, partial P = A^T X with A = W U   (Tc)
//            (pseudo-inverse and complement projector, Sec. 2.2; Eq. 2.16 times dt);
//            dS = Y_2 x_2 A_2^T on the CTAs without rows (all of them where every one has some)
//   2 rows : P_n = sum of the partials, E = X - U P_n (Tc), U' = U + E (double;
//            Euler step, Sec. 2.3), partial C = U'^T W U' (Tc)
//   3 rows : C_n = R^T R and R^{-1} (weighted Cholesky-QR, the reading used to keep Eq. 2.6
//            through the step), by every CTA for the mode of its rows (the same instructions
//            on the same sums; cheaper than one CTA's result through L2 and a barrier);
//            U'' = U' R^{-1} (double), A = W U'' and U'' in Tc
//   4 slabs: (T + dS) x_1 R_1 x_2 R_2, the r_1 x r_2 slabs of the core (double; T x U is left
//            unchanged)
//   5      : x_3 R_3 (x_4 R_4), the r_3 x r_4 fibers; the core and its copy in Tc
//   6 tasks: partial G_n = T_(n) T_(n)^T over column slices (double)
//   7 mode : G_n, G_n^{-1} by Gauss-Jordan (double); sigma^2 (Eq. 2.18) by a float
//            Jacobi warm-started from the previous eigenvectors, then Rayleigh
//            quotients in double
// GB300 issues one double warp-instruction per 64 cycles per SM sub-partition,
// with the same latency: double work is spread over all CTAs where it is a
// throughput cost and kept off the long serial chains where it is a latency cost.
// In the float compute type, C_n = I + D is accumulated in float; R comes from a
// series in D when D is small (as after every regular step) and otherwise from a
// float Cholesky with R^{-1} from one double Newton step on its float inverse.
// Either way R^{-1} R = I to double rounding (the core compensation stays exact)
// while U^T W U = I holds to the accuracy of C_n.
#include "common.cuh"
#include "kernels.h"
#include "small_dev.cuh"
#include "tc_project.h"

namespace tdb {

namespace {

constexpr int LD = kMaxRank;
constexpr int UPD_THREADS = 1024;
constexpr size_t kUpdSmem = 54 * 1024;   // largest phase: the rows of phase 1 in double, 49.3 KB
constexpr int GJ_THREADS = 256;          // threads 0..255 invert G_n by Gauss-Jordan
// Modes with more row tiles than this (more than 1024 points) have their per-tile partial
// sums of P_n and C_n reduced once by the whole grid (reduce_long) instead of by every
// tile's CTA (P_n) or the mode's one CTA (C_n).
constexpr int kTreeTiles = 32;

__device__ __forceinline__ void named_bar(int id, int nthreads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// Order-preserving integer key of a double (larger value, larger key).
__device__ __forceinline__ long long order_key(double v) {
  const long long b = __double_as_longlong(v);
  return b >= 0 ? b : (long long)(b ^ 0x7fffffffffffffffLL);
}

// Packed upper-triangle index e -> (a <= b), e < r (r + 1) / 2, column by column.
__device__ __forceinline__ void tri_index(int e, int* a, int* b) {
  int bb = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
  while ((bb + 1) * (bb + 2) / 2 <= e) ++bb;
  while (bb * (bb + 1) / 2 > e) --bb;
  *b = bb;
  *a = e - bb * (bb + 1) / 2;
}

// ---------------------------------------------------------------------------
// Double Cholesky S = L L^T in place (lower) and L^{-1}, all threads of the CTA
// (the double compute type's Cholesky-QR).
// ---------------------------------------------------------------------------
__device__ bool chol_d(double* S, int r, bool* ok_sh, double* dinv_sh) {
  if (threadIdx.x == 0) *ok_sh = true;
  __syncthreads();
  for (int k = 0; k < r; ++k) {
    if (threadIdx.x == 0) {
      double d = S[k + LD * k];
      if (!(d > 0.0)) { *ok_sh = false; d = 1.0; }
      const double inv = drsqrt(d);
      S[k + LD * k] = d * inv;
      *dinv_sh = inv;
    }
    __syncthreads();
    const double inv = *dinv_sh;
    for (int i = k + 1 + threadIdx.x; i < r; i += blockDim.x) S[i + LD * k] *= inv;
    __syncthreads();
    const int m = r - k - 1;
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
      const int i = k + 1 + e % m, j = k + 1 + e / m;
      if (j <= i) S[i + LD * j] -= S[i + LD * k] * S[j + LD * k];
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < r * r; e += blockDim.x) {
    const int i = e % r, j = e / r;
    if (j > i) S[i + LD * j] = 0.0;
  }
  __syncthreads();
  return *ok_sh;
}

__device__ void trinv_d(const double* L, double* Li, int r, double* dinv) {
  for (int i = threadIdx.x; i < r; i += blockDim.x) dinv[i] = drcp(L[i + LD * i]);
  __syncthreads();
  for (int j = threadIdx.x; j < r; j += blockDim.x) {
    for (int i = 0; i < r; ++i) {
      if (i < j) { Li[i + LD * j] = 0.0; continue; }
      double s = (i == j) ? 1.0 : 0.0;
      for (int k = j; k < i; ++k) s -= L[i + LD * k] * Li[k + LD * j];
      Li[i + LD * j] = s * dinv[i];
    }
  }
  __syncthreads();
}

// ---------------------------------------------------------------------------
// Float Cholesky S = L L^T and Li = L^{-1} by one warp (the float compute type's Cholesky-QR),
// r <= RM, ld LD, in shared memory.  Lane i keeps row i of S, then lane j column j of Li, in
// registers: a step is one shuffle, one reciprocal and independent multiply-adds (working in
// shared memory it waited for a load and a store per entry: 3.2 us at r = 6).
// ---------------------------------------------------------------------------
template <int RM>
__device__ bool chol_inv_warp_f(float* S, float* Li, int r) {
  const int lane = threadIdx.x & 31;
  bool ok = true;
  float a[RM];
#pragma unroll
  for (int j = 0; j < RM; ++j) a[j] = (lane < r && j < r) ? S[lane + LD * j] : 0.f;
#pragma unroll
  for (int k = 0; k < RM; ++k) {
    if (k >= r) break;
    float d = __shfl_sync(0xffffffffu, a[k], k);
    if (!(d > 0.f)) { ok = false; d = 1.f; }
    const float inv = rsqrt_approx(d);
    const float lik = lane > k ? a[k] * inv : 0.f;
#pragma unroll
    for (int j = k + 1; j < RM; ++j) {
      const float ljk = __shfl_sync(0xffffffffu, lik, j);
      if (lane >= j) a[j] = fmaf(-lik, ljk, a[j]);
    }
    a[k] = lane > k ? lik : (lane == k ? d * inv : 0.f);
  }
#pragma unroll
  for (int j = 0; j < RM; ++j)
    if (lane < r && j < r) S[lane + LD * j] = a[j];
  __syncwarp();
  float x[RM];
#pragma unroll
  for (int i = 0; i < RM; ++i) x[i] = i == lane ? 1.f : 0.f;
#pragma unroll
  for (int k = 0; k < RM; ++k) {
    if (k >= r) break;
    if (lane <= k) {
      x[k] = x[k] / S[k + LD * k];
#pragma unroll
      for (int i = k + 1; i < RM; ++i)
        if (i < r) x[i] = fmaf(-S[i + LD * k], x[k], x[i]);
    }
  }
#pragma unroll
  for (int i = 0; i < RM; ++i)
    if (lane < r && i < r) Li[i + LD * lane] = x[i];
  __syncwarp();
  return ok;
}

// ---------------------------------------------------------------------------
// Cyclic Jacobi on a symmetric float matrix (n <= 32, ld LD, shared) by a group of
// JG = 256 threads (gt = index in the group, hardware barrier `bar`), Brent-Luk
// round-robin ordering: eigenvalues end on the diagonal of the returned buffer (A or B) and
// the vectors in V.  Stops when the off-diagonal mass is below tol^2 of the diagonal
// mass, after max_sweeps, or when a sweep after the second no longer halves it
// (the float rounding floor).  red holds >= 16 floats.
//
// A round is one chain (the pair's entries, its rotation, the 2 x 2 block) between barriers;
// every thread forms the two rotations its block needs itself, from the buffer the round
// reads, and writes the block to the other one, so a round has one barrier.  (The rotations
// formed by half the pairs' threads and passed through shared memory: two barriers and 0.5 us
// a round.)  V's entries belong to one thread in a round and stay in place.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void jacobi_pair(int nn, int rd, int k, int& p, int& q) {
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
__device__ __forceinline__ void jacobi_rotation(float app, float aqq, float apq, float thr, float& c, float& s) {
  c = 1.f;
  s = 0.f;
  if (apq != 0.f && apq * apq > thr * thr * fabsf(app * aqq)) {
    // tan of the rotation angle, t = sign(theta) / (|theta| + sqrt(theta^2 + 1)),
    // with approximate reciprocals: c^2 + s^2 = 1 holds whatever t's rounding
    const float theta = (aqq - app) * rcp_approx(2.f * apq);
    const float at = fabsf(theta);
    const float x = fmaf(at, at, 1.f);
    const float root = (at < 1e18f) ? x * rsqrt_approx(x) : at;
    const float t = copysignf(rcp_approx(at + root), theta);
    c = rsqrt_approx(fmaf(t, t, 1.f));
    s = t * c;
  }
}
constexpr int JG = 256;
__device__ float* jacobi_group(float* A, float* B, float* V, int n, int max_sweeps, float tol, float* red, int gt,
                               int bar) {
  const int nn = (n + 1) & ~1, half = nn / 2;
  constexpr int nw = JG >> 5;
  const int gl = gt & 31, gw = gt >> 5;
  for (int e = gt; e < nn * nn; e += JG) {
    const int i = e % nn, j = e / nn;
    if (i >= n || j >= n) A[i + LD * j] = 0.f;
    V[i + LD * j] = (i == j) ? 1.f : 0.f;
  }
  // the block (I, J) and the V entries (i, J) of this thread, fixed for all rounds
  const int bI = gt % half, bJ = gt / half;
  const bool has_b = gt < half * half;
  const int nv = nn * half;
  const int v0 = gt < nv ? gt : -1, v1 = gt + JG < nv ? gt + JG : -1;
  const int vi0 = v0 % nn, vJ0 = v0 / nn, vi1 = v1 % nn, vJ1 = v1 / nn;
  named_bar(bar, JG);
  const float thr = tol * 1e-3f;
  float off_prev = 0.f;
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    float off = 0.f, dia = 0.f;
    for (int e = gt; e < nn * nn; e += JG) {
      const int i = e % nn, j = e / nn;
      const float v = A[i + LD * j];
      if (i == j) dia += v * v; else off += v * v;
    }
    off = warp_sum(off);
    dia = warp_sum(dia);
    if (gl == 0) { red[gw] = off; red[nw + gw] = dia; }
    named_bar(bar, JG);
    off = 0.f;
    dia = 0.f;
    for (int w = 0; w < nw; ++w) { off += red[w]; dia += red[nw + w]; }
    named_bar(bar, JG);
    if (off <= tol * tol * dia || dia == 0.f) break;
    if (sweep >= 2 && off > 0.5f * off_prev) break;
    off_prev = off;
    auto rotation = [&](int p, int q, float& c, float& s) {
      jacobi_rotation(A[p + LD * p], A[q + LD * q], A[p + LD * q], thr, c, s);
    };
    auto turn = [&](int rd, int i, int J) {              // V's entry (i, pair J)
      int p, q;
      jacobi_pair(nn, rd, J, p, q);
      float c, s;
      rotation(p, q, c, s);
      const float vp = V[i + LD * p], vq = V[i + LD * q];
      V[i + LD * p] = c * vp - s * vq;
      V[i + LD * q] = s * vp + c * vq;
    };
    for (int rd = 0; rd < nn - 1; ++rd) {
      if (has_b) {
        int pI, qI, pJ, qJ;
        jacobi_pair(nn, rd, bI, pI, qI);
        jacobi_pair(nn, rd, bJ, pJ, qJ);
        const float b00 = A[pI + LD * pJ], b01 = A[pI + LD * qJ], b10 = A[qI + LD * pJ], b11 = A[qI + LD * qJ];
        float cI, sI, cJ, sJ;
        rotation(pI, qI, cI, sI);
        rotation(pJ, qJ, cJ, sJ);
        const float c00 = cJ * b00 - sJ * b01, c01 = sJ * b00 + cJ * b01;
        const float c10 = cJ * b10 - sJ * b11, c11 = sJ * b10 + cJ * b11;
        B[pI + LD * pJ] = cI * c00 - sI * c10;
        B[pI + LD * qJ] = cI * c01 - sI * c11;
        B[qI + LD * pJ] = sI * c00 + cI * c10;
        B[qI + LD * qJ] = sI * c01 + cI * c11;
      }
      if (v0 >= 0) turn(rd, vi0, vJ0);
      if (v1 >= 0) turn(rd, vi1, vJ1);
      named_bar(bar, JG);
      float* t = A;
      A = B;
      B = t;
    }
  }
  return A;
}

// Gauss-Jordan inversion of the SPD matrix in A0 (r x r, ld LD, shared) by the
// threads [0, nthr) with hardware barrier `bar`, no pivoting (the pivots are the
// positive Schur-complement diagonals).  Step k reads one buffer and writes the
// other, so a step needs one barrier; returns the buffer holding the inverse.  The
// reciprocal of the next pivot is formed once, by the thread that updates that
// diagonal entry, into ipk[(k+1) & 1] (FP64 issues one warp-instruction per 64 cycles
// per SM sub-partition, so every thread forming it would cost the step more than the
// update itself).  *ok is false if a pivot is not a positive finite number.
__device__ double* gj_inverse(double* A0, double* A1, int r, int nthr, int bar, bool* ok, double* ipk, int* bad) {
  const int tid = threadIdx.x;
  double* cur = A0;
  double* nxt = A1;
  auto pivot_rcp = [&](double p, int slot) {
    const int hi = __double2hiint(p);
    if (hi <= 0 || ((hi >> 20) & 0x7ff) == 0x7ff) { *bad = 1; p = 1.0; }
    ipk[slot] = drcp(p);
  };
  if (tid == 0) {
    *bad = 0;
    pivot_rcp(cur[0], 0);
  }
  // this thread's entries (i, j), the same in every step (packed i | j << 8, -1 none)
  constexpr int EPT = LD * LD / GJ_THREADS;
  int ent[EPT];
#pragma unroll
  for (int u = 0; u < EPT; ++u) {
    const int e = tid + nthr * u;
    ent[u] = e < r * r ? ((e % r) | ((e / r) << 8)) : -1;
  }
  named_bar(bar, nthr);
  for (int k = 0; k < r; ++k) {
    const double ip = ipk[k & 1];
#pragma unroll
    for (int u = 0; u < EPT; ++u) {
      if (ent[u] < 0) continue;
      const int i = ent[u] & 255, j = ent[u] >> 8;
      const double akj = (j == k) ? ip : cur[k + LD * j] * ip;     // row k after the step
      const double v = (i == k) ? akj : (j == k ? 0.0 : cur[i + LD * j]) - cur[i + LD * k] * akj;
      nxt[i + LD * j] = v;
      if (i == k + 1 && j == k + 1) pivot_rcp(v, (k + 1) & 1);
    }
    named_bar(bar, nthr);
    double* t = cur;
    cur = nxt;
    nxt = t;
  }
  *ok = *bad == 0;
  return cur;
}

// Bounded grid barrier; every CTA is resident (cooperative launch, <= 1 CTA per SM).
// The counter (zeroed at the start of the step) only grows: the k-th barrier (k from 1)
// waits for k * nblocks arrivals.  Release on arrival and acquire on the spin order
// the CTA's writes before and its reads after the barrier.
__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release_gpu(unsigned* p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
constexpr long long kGridWaitCycles = 4000000000ll;   // ~2 s at 2 GHz
__device__ __forceinline__ bool grid_sync(unsigned* count, unsigned k, unsigned nblocks, unsigned* flags,
                                          volatile int* abort_sh, long long limit = kGridWaitCycles) {
  __syncthreads();
  if (threadIdx.x == 0) {
    red_release_gpu(count, 1u);
    const unsigned target = k * nblocks;
    const long long t0 = clock64();
    unsigned it = 0;
    // one load per poll; the clock and another CTA's timeout flag every 32nd
    while (ld_acquire_gpu(count) < target) {
      if ((++it & 31) == 0 && (clock64() - t0 > limit || (ld_acquire_gpu(flags) & kFlagTimeout))) {
        atomicOr(flags, kFlagTimeout);
        *abort_sh = 1;
        break;
      }
    }
  }
  __syncthreads();
  return *abort_sh == 0;
}

// Profiling: CTA 0 reads the global timer at the start, after every grid barrier
// and at its end into shared memory; at the end it adds the phase durations to
// st[16 + k] (nanoseconds summed over launches; st null when profiling is off).
__device__ __forceinline__ void stamp(unsigned long long* sh, const unsigned long long* st, int k) {
  if (st && blockIdx.x == 0 && threadIdx.x == 0) {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    sh[k] = t;
  }
}
__device__ __forceinline__ void stamp_flush(const unsigned long long* sh, unsigned long long* st, int nst) {
  if (st && blockIdx.x == 0 && threadIdx.x == 0)
    for (int k = 1; k <= nst; ++k) atomicAdd(&st[16 + k - 1], sh[k] - sh[k - 1]);
}

}  // namespace

// ---------------------------------------------------------------------------
// Gram refresh, shared by the fused update and the standalone launches.
// ---------------------------------------------------------------------------

// Partial G_n = T_(n) T_(n)^T over column slice `sp` of mode n: the slice is staged
// in shared memory 32 columns at a time; one thread per upper-triangle entry, its sum in
// CH interleaved chains (4 in the float types: a chain of 32 dependent double products is 2 us).
template <int CH>
__device__ void gram_partial(const ModeDesc& d, const double* T, double* gpart, int gsplit, int n, int sp,
                             double (*S)[33]) {
  const int r = d.r[n];
  const int64_t L = prod_r_below(d, n), Q = prod_r_above(d, n);
  const int64_t ncol = L * Q;
  const int64_t c0 = ncol * sp / gsplit, c1 = ncol * (sp + 1) / gsplit;
  const int ntri = r * (r + 1) / 2;
  int ta = 0, tb = 0;
  if ((int)threadIdx.x < ntri) tri_index(threadIdx.x, &ta, &tb);
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  double sum[CH];
#pragma unroll
  for (int u = 0; u < CH; ++u) sum[u] = 0.0;
  for (int64_t cb = c0; cb < c1; cb += 32) {
    const int64_t c = cb + tx;
    double v = 0.0;
    if (c < c1 && ty < r) {
      const int64_t l = c % L, q = c / L;
      v = __ldcg(&T[l + L * (ty + (int64_t)r * q)]);
    }
    S[ty][tx] = v;
    __syncthreads();
    if ((int)threadIdx.x < ntri) {
#pragma unroll
      for (int x = 0; x < 32; ++x) sum[x % CH] = fma(S[ta][x], S[tb][x], sum[x % CH]);
    }
    __syncthreads();
  }
  double s = sum[0];
#pragma unroll
  for (int u = 1; u < CH; ++u) s += sum[u];
  if ((int)threadIdx.x < ntri) gpart[((int64_t)n * gsplit + sp) * LD * LD + ta + LD * tb] = s;
}

// Mode n: sum the partials into G_n; G_n^{-1} by Gauss-Jordan (threads 0..255)
// while threads 256..511 run the float Jacobi on Vp^T (G / scale) Vp (Vp the previous
// eigenvectors, identity when cold); then Rayleigh quotients v^T G v / v^T v in
// double, sorted descending by an integer key; the sorted eigenvectors become the
// next warm start.  One CTA of UPD_THREADS threads; smraw holds >= 50 KB.
__device__ __noinline__ void gram_finish(const ModeDesc& d, int n, const double* gpart, int gsplit, double* Gout,
                                         double* Ginv, float* Ginvf, double* sig2, float* Vprev, int warm,
                                         unsigned* flags, unsigned char* smraw) {
  const int r = d.r[n];
  double* G = (double*)smraw;          // LD*LD
  double* Ai = G + LD * LD;            // LD*LD: Gauss-Jordan buffers, then G W
  double* Ai2 = Ai + LD * LD;          // LD*LD
  double* lam = Ai2 + LD * LD;         // LD
  float* Gf = (float*)(lam + LD);      // LD*LD: G / scale in float
  float* Vps = Gf + LD * LD;           // LD*LD: previous eigenvectors
  float* Af = Vps + LD * LD;           // LD*LD
  float* Vf = Af + LD * LD;            // LD*LD  (Af and Vf later hold W in double)
  float* Wf = Vf + LD * LD;            // LD*LD
  float* Bf = Wf + LD * LD;            // LD*LD: the Jacobi's other buffer
  float* red = Bf + LD * LD;           // 64
  int* slot = (int*)(red + 64);        // LD
  double* GW = Ai;
  double* Wd = (double*)Af;
  __shared__ int bad_sh, gjbad_sh;
  __shared__ float scale_sh;
  __shared__ double ipk_sh[2];
  const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
  float* Vp = Vprev + (int64_t)n * LD * LD;
  if (tid == 0) bad_sh = 0;
  for (int e = tid; e < LD * LD; e += blockDim.x) {
    const int ra = e % LD, rb = e / LD;
    double s = 0.0;
    if (ra < r && rb < r) {
      const int aa = ra <= rb ? ra : rb, bb = ra <= rb ? rb : ra;
      const double* src = gpart + (int64_t)n * gsplit * LD * LD + aa + LD * bb;
#pragma unroll 8
      for (int k = 0; k < gsplit; ++k) s += __ldcg(&src[(int64_t)k * LD * LD]);
    }
    G[e] = s;
    Ai[e] = s;
    Vps[e] = (warm && ra < r && rb < r) ? Vp[e] : 0.f;
  }
  __syncthreads();
  if (wid == 0) {
    float m = 0.f;
    for (int k = lane; k < r; k += 32) m = fmaxf(m, (float)G[k + LD * k]);
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) scale_sh = m > 0.f ? 1.f / m : 1.f;
  }
  __syncthreads();
  for (int e = tid; e < r * r; e += blockDim.x) {
    const int a = e % r, b = e / r;
    Gf[a + LD * b] = (float)G[a + LD * b] * scale_sh;
  }
  __syncthreads();
  __shared__ double* inv_sh;
  if (tid < GJ_THREADS) {
    bool good;
    double* res = gj_inverse(Ai, Ai2, r, GJ_THREADS, 1, &good, ipk_sh, &gjbad_sh);
    if (tid == 0) {
      inv_sh = res;
      if (!good) bad_sh = 1;
    }
  } else if (tid < GJ_THREADS + JG) {
    const int gt = tid - GJ_THREADS;
    if (warm) {
      for (int e = gt; e < r * r; e += JG) {             // Wf = (G / scale) Vp
        const int i = e % r, b = e / r;
        float s = 0.f;
        for (int j = 0; j < r; ++j) s = fmaf(Gf[i + LD * j], Vps[j + LD * b], s);
        Wf[i + LD * b] = s;
      }
      named_bar(2, JG);
      for (int e = gt; e < r * r; e += JG) {             // Af = Vp^T Wf
        const int a = e % r, b = e / r;
        float s = 0.f;
        for (int i = 0; i < r; ++i) s = fmaf(Vps[i + LD * a], Wf[i + LD * b], s);
        Af[a + LD * b] = s;
      }
    } else {
      for (int e = gt; e < r * r; e += JG) {
        const int a = e % r, b = e / r;
        Af[a + LD * b] = Gf[a + LD * b];
      }
    }
    named_bar(2, JG);
    jacobi_group(Af, Bf, Vf, r, warm ? 2 : 30, 1e-6f, red, gt, 2);
    for (int e = gt; e < r * r; e += JG) {               // eigenvectors in the original basis
      const int a = e % r, b = e / r;
      float s = Vf[a + LD * b];
      if (warm) {
        s = 0.f;
        for (int k = 0; k < r; ++k) s = fmaf(Vps[a + LD * k], Vf[k + LD * b], s);
      }
      Wf[a + LD * b] = s;
    }
  }
  __syncthreads();
  if (bad_sh && tid == 0) atomicOr(flags, kFlagCholGram);
  for (int e = tid; e < LD * LD; e += blockDim.x) {
    const int a = e % LD, b = e / LD;
    const bool in = a < r && b < r;
    const double gi = in ? inv_sh[e] : 0.0;
    Gout[(int64_t)n * LD * LD + e] = G[e];
    Ginv[(int64_t)n * LD * LD + e] = gi;
    if (Ginvf) Ginvf[(int64_t)n * LD * LD + e] = in ? (float)gi : 0.f;
  }
  __syncthreads();
  for (int e = tid; e < r * r; e += blockDim.x) {
    const int a = e % r, b = e / r;
    Wd[a + LD * b] = (double)Wf[a + LD * b];
  }
  __syncthreads();
  // Rayleigh quotients: GW = G W, then warp j reduces column j
  for (int e = tid; e < r * r; e += blockDim.x) {
    const int i = e % r, j = e / r;
    double s = 0.0;
    for (int k = 0; k < r; ++k) s = fma(G[i + LD * k], Wd[k + LD * j], s);
    GW[i + LD * j] = s;
  }
  __syncthreads();
  if (wid < r) {
    const int j = wid;
    double num = 0.0, den = 0.0;
    if (lane < r) {
      const double v = Wd[lane + LD * j];
      num = v * GW[lane + LD * j];
      den = v * v;
    }
    num = warp_sum(num);
    den = warp_sum(den);
    if (lane == 0) lam[j] = den > 0.0 ? num * drcp(den) : 0.0;
  }
  __syncthreads();
  if (tid < r) {                                         // descending rank by integer keys
    const long long kj = order_key(lam[tid]);
    int rank = 0;
    for (int k = 0; k < r; ++k) {
      const long long kk = order_key(lam[k]);
      rank += (kk > kj) || (kk == kj && k < tid);
    }
    slot[tid] = rank;
    sig2[(int64_t)n * LD + rank] = lam[tid];
  } else if (tid < LD) {
    sig2[(int64_t)n * LD + tid] = 0.0;
  }
  __syncthreads();
  for (int e = tid; e < r * r; e += blockDim.x) {
    const int i = e % r, j = e / r;
    Vp[i + LD * slot[j]] = Wf[i + LD * j];
  }
}

// ---------------------------------------------------------------------------
// Row-tile phases
// ---------------------------------------------------------------------------

// N consecutive values (16-byte aligned) from shared memory
template <typename Tc, int N>
__device__ __forceinline__ void lds_vec(const Tc* p, Tc* v) {
  constexpr int per = 16 / sizeof(Tc);
#pragma unroll
  for (int i = 0; i < N / per; ++i) {
    if constexpr (sizeof(Tc) == 4) {
      const float4 t = reinterpret_cast<const float4*>(p)[i];
      v[4 * i] = t.x; v[4 * i + 1] = t.y; v[4 * i + 2] = t.z; v[4 * i + 3] = t.w;
    } else {
      const double2 t = reinterpret_cast<const double2*>(p)[i];
      v[2 * i] = t.x; v[2 * i + 1] = t.y;
    }
  }
}

// Phase 1 on one tile of mode n: M = Y_(n) T_(n)^T, X = M G^{-1}, partial P = A^T X.  The
// columns come in chunks of CW, all of a chunk's loads in flight at once and the next chunk's
// behind the products (32 columns at a time paid the L2 latency up to 19 times), read back as
// 16-byte vectors.
template <typename Tc>
__device__ void rows_mxp(const UpdArgs& a, int n, int64_t i0, int tile, unsigned char* sm) {
  constexpr int CW = sizeof(Tc) == 4 ? 128 : 64, CPT = CW / 32, LDC = CW + 16 / (int)sizeof(Tc);
  constexpr int VN = 16 / sizeof(Tc);
  const ModeDesc& d = a.d;
  const int r = d.r[n];
  const int64_t N = d.N[n];
  const int li = threadIdx.x & 31, ca = threadIdx.x >> 5;
  const int64_t i = i0 + li;
  Tc (*Ysh)[LDC] = (Tc(*)[LDC])sm;
  Tc (*Tsh)[LDC] = Ysh + 32;
  Tc (*Msh)[33] = (Tc(*)[33])(Tsh + 32);
  Tc* Gi = (Tc*)(Msh + 32);
  const unsigned L = (unsigned)prod_r_below(d, n), ncol = L * (unsigned)prod_r_above(d, n);
  const Tc* Y = (const Tc*)a.Y[n];
  const Tc* Tm = (const Tc*)a.Tcore;
  if (sizeof(Tc) == 8) {
    for (int e = threadIdx.x; e < LD * LD; e += blockDim.x) Gi[e] = (Tc)a.Ginv[(int64_t)n * LD * LD + e];
  } else {
    for (int e = threadIdx.x; e < LD * LD; e += blockDim.x) Gi[e] = (Tc)a.Ginvf[(int64_t)n * LD * LD + e];
  }
  Tc s = Tc(0);
  // staging: for L == 1 the rows of Y_(n) (and the ranks of T_(n)) are contiguous, so
  // lanes run along rows; otherwise along columns
  const bool rows_fast = (L == 1);
  const int u = threadIdx.x & 31, v = threadIdx.x >> 5;
  const int srow = rows_fast ? u : v, scol = rows_fast ? v : u;
  const bool yin = i0 + srow < N, tin = srow < r;
  Tc vy[CPT], vt[CPT];
  auto fetch = [&](unsigned c0) {
#pragma unroll
    for (int k = 0; k < CPT; ++k) {
      const unsigned c = c0 + scol + 32 * k;
      vy[k] = Tc(0);
      vt[k] = Tc(0);
      if (c < ncol) {
        const unsigned q = c / L, l = c - q * L;
        if (yin) vy[k] = Y[l + (size_t)L * (i0 + srow + (size_t)N * q)];
        if (tin) vt[k] = Tm[l + (size_t)L * (srow + (size_t)r * q)];
      }
    }
  };
  fetch(0);
  for (unsigned c0 = 0; c0 < ncol; c0 += CW) {
#pragma unroll
    for (int k = 0; k < CPT; ++k) {
      Ysh[srow][scol + 32 * k] = vy[k];
      Tsh[srow][scol + 32 * k] = vt[k];
    }
    __syncthreads();
    if (c0 + CW < ncol) fetch(c0 + CW);
    if (ca < r) {
      const int nx = (int)min((unsigned)CW, (ncol - c0 + 31) & ~31u);     // (zeros past ncol)
#pragma unroll 4
      for (int x = 0; x < nx; x += VN) {
        Tc y[VN], t[VN];
        lds_vec<Tc, VN>(&Ysh[li][x], y);
        lds_vec<Tc, VN>(&Tsh[ca][x], t);
#pragma unroll
        for (int w = 0; w < VN; ++w) s += y[w] * t[w];
      }
    }
    __syncthreads();
  }
  if (ca < r) Msh[li][ca] = s;
  Tc (*Ash)[33] = (Tc(*)[33])sm;
  Tc (*Xsh)[33] = Ash + 32;
  Ash[li][ca] = (ca < r && i < N) ? ((const Tc*)a.A[n])[i + N * ca] : Tc(0);
  __syncthreads();
  Tc x = Tc(0);
  if (ca < r && i < N) {
    for (int b = 0; b < r; ++b) x += Msh[li][b] * Gi[b + LD * ca];
    ((Tc*)a.X[n])[i + N * ca] = x;
  }
  Xsh[li][ca] = x;
  __syncthreads();
  if ((int)threadIdx.x < r * r) {
    const int ra = threadIdx.x % r, rb = threadIdx.x / r;
    Tc acc = Tc(0);
#pragma unroll 8
    for (int t = 0; t < 32; ++t) acc += Ash[t][ra] * Xsh[t][rb];
    ((Tc*)a.part)[((int64_t)n * a.ntile + tile) * LD * LD + ra + LD * rb] = acc;
  }
  __syncthreads();
}

// Phase 2 on one tile of mode n: P_n, E = X - U P_n, U' = U + E (Heun's second stage:
// U' = (U0 + U + E) / 2; the midpoint scheme's second stage: U' = U0 + E), partial
// C = U'^T W U'.
template <typename Tc>
__device__ void rows_u1(const UpdArgs& a, int n, int64_t i0, int tile, unsigned char* sm) {
  const ModeDesc& d = a.d;
  const int r = d.r[n];
  const int64_t N = d.N[n];
  const int li = threadIdx.x & 31, ca = threadIdx.x >> 5;
  const int64_t i = i0 + li;
  Tc* Psh = (Tc*)sm;                         // LD*LD
  Tc (*Ush)[33] = (Tc(*)[33])(Psh + LD * LD);
  Tc (*Wsh)[33] = Ush + 32;                  // U' W
  const Tc wi = i < N ? (Tc)a.w[n][i] : Tc(0);
  const Tc* part = (const Tc*)a.part;
  const int nt = (int)((N + 31) / 32);
  {
    const int e = threadIdx.x, ra = e % LD, rb = e / LD;
    Tc s = Tc(0);
    if (ra < r && rb < r) {
      if (nt > kTreeTiles) {
        s = __ldcg(&((const Tc*)a.red)[(int64_t)n * LD * LD + e]);
      } else {
        const Tc* src = part + (int64_t)n * a.ntile * LD * LD + e;
#pragma unroll 8
        for (int t = 0; t < nt; ++t) s += __ldcg(&src[(int64_t)t * LD * LD]);
      }
    }
    Psh[e] = s;
  }
  Ush[li][ca] = (ca < r && i < N) ? ((const Tc*)a.Uc[n])[i + N * ca] : Tc(0);
  __syncthreads();
  Tc upc = Tc(0);
  if (ca < r && i < N) {
    Tc e = __ldcg(&((const Tc*)a.X[n])[i + N * ca]);
    for (int b = 0; b < r; ++b) e -= Ush[li][b] * Psh[b + LD * ca];
    const int64_t ix = i + N * ca;
    const double up = !a.T0             ? a.U[n][ix] + (double)e
                      : a.combine == 2 ? a.U0[n][ix] + (double)e
                                       : 0.5 * ((a.U[n][ix] + a.U0[n][ix]) + (double)e);
    a.Up[n][i + N * ca] = up;
    upc = (Tc)up;
  }
  __syncthreads();
  Ush[li][ca] = upc;
  Wsh[li][ca] = upc * wi;
  __syncthreads();
  if ((int)threadIdx.x < r * r) {
    const int ra = threadIdx.x % r, rb = threadIdx.x / r;
    Tc acc = Tc(0);
#pragma unroll 8
    for (int t = 0; t < 32; ++t) acc += Wsh[t][ra] * Ush[t][rb];
    ((Tc*)a.part)[(int64_t)a.d.p * a.ntile * LD * LD + ((int64_t)n * a.ntile + tile) * LD * LD + ra + LD * rb] = acc;
  }
  __syncthreads();
}

// Phases 1b / 2b, only for modes with more than kTreeTiles row tiles: the per-tile
// partials of P_n (which = 0) or C_n (which = 1) summed by the whole grid, a warp per
// entry, its lanes over every 32nd tile, then a butterfly of shuffles (the same order on
// every run).  Results go to red[which][n], read by every tile of phase 2 (P_n) or by
// the Cholesky-QR of phase 3 (C_n).
template <typename Tc>
__device__ void reduce_long(const UpdArgs& a, int which, unsigned bid, unsigned nb) {
  const ModeDesc& d = a.d;
  const int lane = threadIdx.x & 31;
  const int64_t gw = (int64_t)bid * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int64_t nw = (int64_t)nb * (blockDim.x >> 5);
  const Tc* part = (const Tc*)a.part + (int64_t)which * d.p * a.ntile * LD * LD;
  Tc* red = (Tc*)a.red + (int64_t)which * kMaxModes * LD * LD;
  for (int64_t task = gw; task < (int64_t)d.p * LD * LD; task += nw) {
    const int n = (int)(task / (LD * LD)), e = (int)(task % (LD * LD));
    const int nt = (int)((d.N[n] + 31) / 32);
    const int r = d.r[n], ra = e % LD, rb = e / LD;
    if (nt <= kTreeTiles || ra >= r || rb >= r) continue;     // the same for the whole warp
    const Tc* src = part + (int64_t)n * a.ntile * LD * LD + e;
    Tc s = Tc(0);
    for (int t = lane; t < nt; t += 32) s += __ldcg(&src[(int64_t)t * LD * LD]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) red[(int64_t)n * LD * LD + e] = s;
  }
}

// Phase 3 for mode n: C_n from the partials, R (upper, C = R^T R) and R^{-1} into the first
// two LD x LD doubles of sm (R, then R^{-1}); 24 KB of scratch after them.  Every CTA with
// rows of the mode forms the same factors; `flag` only on one of them.
template <typename Tc>
__device__ void mode_cholqr(const UpdArgs& a, int n, unsigned char* sm, bool flag) {
  const ModeDesc& d = a.d;
  const int r = d.r[n];
  const int nt = (int)((d.N[n] + 31) / 32);
  const Tc* part = (const Tc*)a.part + (int64_t)d.p * a.ntile * LD * LD + (int64_t)n * a.ntile * LD * LD;
  double* Rs = (double*)sm;
  double* Ris = Rs + LD * LD;
  unsigned char* scr = (unsigned char*)(Ris + LD * LD);
  __shared__ bool ok_sh;
  __shared__ double dinv_sh;
  const int e = threadIdx.x, ra = e % LD, rb = e / LD;      // (UPD_THREADS == LD * LD)
  if (!a.reorth) {
    Rs[e] = Ris[e] = ra == rb ? 1.0 : 0.0;
    __syncthreads();
    return;
  }
  Tc c = Tc(0);
  if (ra < r && rb < r) {
    if (nt > kTreeTiles)
      c = __ldcg(&((const Tc*)a.red)[(int64_t)(kMaxModes + n) * LD * LD + e]);
    else
#pragma unroll 8
      for (int t = 0; t < nt; ++t) c += __ldcg(&part[(int64_t)t * LD * LD + e]);
  }
  if constexpr (sizeof(Tc) == 8) {
    double* C = (double*)scr;
    double* Li = C + LD * LD;
    double* dinv = Li + LD * LD;
    C[e] = c;
    __syncthreads();
    if (!chol_d(C, r, &ok_sh, &dinv_sh) && threadIdx.x == 0 && flag) atomicOr(a.flags, kFlagCholQR);
    trinv_d(C, Li, r, dinv);
    Rs[e] = (ra < r && rb < r) ? C[rb + LD * ra] : 0.0;     // R = L^T
    Ris[e] = (ra < r && rb < r) ? Li[rb + LD * ra] : 0.0;   // R^{-1} = L^{-T}
  } else {
    float* Cf = (float*)scr;                // LD*LD
    float* F1 = Cf + LD * LD;               // LD*LD
    __shared__ int fmax_sh;
    if (threadIdx.x == 0) fmax_sh = 0;
    // C = I + D with D small after a step: R = I + F, F = Phi(D - F1^T F1), F1 = Phi(D),
    // Phi = upper triangle with the diagonal halved (R^T R = C up to O(|D|^3)), and
    // R^{-1} = I - F + F^2 - F^3 + F^4 (R R^{-1} = I + F^5).  Taken when max |F1| <= 2^-14,
    // so that |F^5| < 4e-14 for r <= 32.
    const bool up = ra <= rb && rb < r;
    const float f1 = up ? (ra == rb ? 0.5f * (c - 1.f) : c) : 0.f;
    Cf[e] = c;
    F1[e] = f1;
    // this thread's entry of the packed upper triangle (the products below are triangular and
    // end in double, which a warp without an entry must not issue)
    const int ntri = r * (r + 1) / 2;
    int ia = 0, jb = 0;
    if (e < ntri) tri_index(e, &ia, &jb);
    __syncthreads();
    {
      float m = fabsf(f1);
      m = (m == m) ? m : 3.0e38f;              // a NaN takes the Cholesky path, which flags it
      for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      if ((threadIdx.x & 31) == 0 && m > 0.f) atomicMax(&fmax_sh, __float_as_int(m));
    }
    __syncthreads();
    if (__int_as_float(fmax_sh) <= 6.103515625e-05f) {
      float* Fs = F1 + LD * LD;                // LD*LD: F
      float* F2 = Fs + LD * LD;                // LD*LD: F^2
      Rs[e] = Ris[e] = 0.0;
      float f = 0.f, f2 = 0.f;
      if (e < ntri) {                          // F = Phi(D - F1^T F1)
        float q = 0.f;
        for (int k = 0; k <= ia; ++k) q = fmaf(F1[k + LD * ia], F1[k + LD * jb], q);
        f = (ia == jb) ? F1[ia + LD * jb] - 0.5f * q : Cf[ia + LD * jb] - q;
        Fs[ia + LD * jb] = f;
      }
      __syncthreads();
      if (e < ntri) {
        for (int k = ia; k <= jb; ++k) f2 = fmaf(Fs[ia + LD * k], Fs[k + LD * jb], f2);
        F2[ia + LD * jb] = f2;
      }
      __syncthreads();
      if (e < ntri) {
        float f3 = 0.f, f4 = 0.f;
        for (int k = ia; k <= jb; ++k) {
          f3 = fmaf(F2[ia + LD * k], Fs[k + LD * jb], f3);
          f4 = fmaf(F2[ia + LD * k], F2[k + LD * jb], f4);
        }
        const double id = ia == jb ? 1.0 : 0.0, fd = (double)f;
        Rs[ia + LD * jb] = id + fd;
        Ris[ia + LD * jb] = (((id - fd) + (double)f2) - (double)f3) + (double)f4;
      }
    } else {
      float* Lif = F1;                         // LD*LD
      double* Z0 = (double*)(F1 + LD * LD);    // LD*LD
      double* E = Z0 + LD * LD;                // LD*LD
      if (threadIdx.x < 32) {
        const bool good = r <= 8 ? chol_inv_warp_f<8>(Cf, Lif, r)
                                 : (r <= 16 ? chol_inv_warp_f<16>(Cf, Lif, r) : chol_inv_warp_f<32>(Cf, Lif, r));
        if (!good && threadIdx.x == 0 && flag) atomicOr(a.flags, kFlagCholQR);
      }
      Rs[e] = Ris[e] = Z0[e] = 0.0;
      __syncthreads();
      if (e < ntri) {
        Rs[ia + LD * jb] = (double)Cf[jb + LD * ia];            // R0 = L^T (upper)
        Z0[ia + LD * jb] = (double)Lif[jb + LD * ia];           // Z0 = L^{-T}, float accurate
      }
      __syncthreads();
      // one Newton step in double: Z1 = Z0 + Z0 (I - R0 Z0); all three are upper triangular
      if (e < ntri) {
        double x = (ia == jb) ? 1.0 : 0.0;
        for (int k = ia; k <= jb; ++k) x = fma(-Rs[ia + LD * k], Z0[k + LD * jb], x);
        E[ia + LD * jb] = x;
      }
      __syncthreads();
      if (e < ntri) {
        double z = Z0[ia + LD * jb];
        for (int k = ia; k <= jb; ++k) z = fma(Z0[ia + LD * k], E[k + LD * jb], z);
        Ris[ia + LD * jb] = z;
      }
    }
  }
  __syncthreads();
}

// Phase 3 on one tile of mode n: U'' = U' R^{-1}, A = W U'' and U'' in the compute type.
template <typename Tc>
__device__ void rows_u2(const UpdArgs& a, int n, int64_t i0, const double* Ris, unsigned char* scr) {
  const ModeDesc& d = a.d;
  const int r = d.r[n];
  const int64_t N = d.N[n];
  const int li = threadIdx.x & 31, ca = threadIdx.x >> 5;
  const int64_t i = i0 + li;
  double (*Ush)[LD + 1] = (double(*)[LD + 1])scr;
  if (ca < r) Ush[li][ca] = (i < N) ? __ldcg(&a.Up[n][i + N * ca]) : 0.0;
  __syncthreads();
  if (ca < r && i < N) {
    double s = 0.0;
    for (int b = 0; b <= ca; ++b) s = fma(Ush[li][b], Ris[b + LD * ca], s);
    a.U[n][i + N * ca] = s;
    ((Tc*)a.A[n])[i + N * ca] = (Tc)(a.w[n][i] * s);
    ((Tc*)a.Uc[n])[i + N * ca] = (Tc)s;
  }
  __syncthreads();
}

// Phase 4: dst = (T + dS) x_1 R_1 x_2 R_2 (Heun's second stage: ((T0 + T + dS) / 2), the
// midpoint scheme's: (T0 + dS)), slab by slab: r_1 x r_2 entries at fixed other indices, F
// slabs at a time staged in shared memory, F chosen so that every CTA of the grid has some.
// With two modes the one slab is the core: it is read whole before it is written.
template <typename Tc>
__device__ void core_12(const UpdArgs& a, unsigned char* sm, unsigned bid, unsigned nb) {
  const ModeDesc& d = a.d;
  const int r1 = d.r[0], r2 = d.r[1], ns = r1 * r2;
  const int64_t nslab = prod_r_above(d, 1);
  const int64_t per_cta = (nslab + nb - 1) / nb;
  const int F = (int)(per_cta < UPD_THREADS / ns ? per_cta : UPD_THREADS / ns);
  if (bid * (int64_t)F >= nslab) return;
  double* R1 = (double*)sm;             // LD*LD each
  double* R2 = R1 + LD * LD;
  double* Xs = R2 + LD * LD;            // F slabs <= UPD_THREADS
  double* Ys = Xs + UPD_THREADS;
  R1[threadIdx.x] = __ldcg(&a.R[threadIdx.x]);
  R2[threadIdx.x] = __ldcg(&a.R[LD * LD + threadIdx.x]);
  const Tc* dS = (const Tc*)a.dS;
  const int t = threadIdx.x, fl = t / ns, e = t - fl * ns, i = e % r1, j = e / r1;
  for (int64_t f0 = bid * (int64_t)F; f0 < nslab; f0 += (int64_t)nb * F) {
    const bool act = fl < F && f0 + fl < nslab;
    const int64_t idx = (f0 + fl) * ns + e;
    if (act) {
      if (a.T0 && a.combine == 2) Xs[t] = a.T0[idx] + (double)dS[idx];
      else if (a.T0) Xs[t] = 0.5 * ((a.T[idx] + a.T0[idx]) + (double)dS[idx]);
      else Xs[t] = a.T[idx] + (double)dS[idx];
    }
    __syncthreads();
    if (act) {
      double s = 0.0;
      for (int k = i; k < r1; ++k) s = fma(R1[i + LD * k], Xs[fl * ns + k + r1 * j], s);
      Ys[t] = s;
    }
    __syncthreads();
    if (act) {
      double s = 0.0;
      for (int k = j; k < r2; ++k) s = fma(R2[j + LD * k], Ys[fl * ns + i + r1 * k], s);
      if (d.p == 2) {
        a.T[idx] = s;
        if (sizeof(Tc) == 4) ((float*)a.Tcore)[idx] = (float)s;
      } else {
        a.T2[idx] = s;
      }
    }
  }
}

// Phase 5: T = T2 x_3 R_3 (x_4 R_4) and its copy in the compute type, by r_3 x r_4 fibers (the
// entries at fixed first two indices), F at a time, neighbouring fibers on neighbouring threads.
template <typename Tc>
__device__ void core_34(const UpdArgs& a, unsigned char* sm, unsigned bid, unsigned nb) {
  const ModeDesc& d = a.d;
  const int r3 = d.r[2], r4 = d.p == 4 ? d.r[3] : 1, nf = r3 * r4;
  const int64_t L = prod_r_below(d, 2);
  const int64_t per_cta = (L + nb - 1) / nb;
  const int F = (int)(per_cta < UPD_THREADS / nf ? per_cta : UPD_THREADS / nf);
  if (bid * (int64_t)F >= L) return;
  double* R3 = (double*)sm;
  double* R4 = R3 + LD * LD;
  double* Xs = R4 + LD * LD;            // F fibers <= UPD_THREADS, element (c, d) of fiber f at f + F (c + r3 d)
  double* Ys = Xs + UPD_THREADS;
  R3[threadIdx.x] = __ldcg(&a.R[2 * LD * LD + threadIdx.x]);
  if (d.p == 4) R4[threadIdx.x] = __ldcg(&a.R[3 * LD * LD + threadIdx.x]);
  const int t = threadIdx.x, fl = t % F, e = t / F, c = e % r3, dd = e / r3;
  for (int64_t f0 = bid * (int64_t)F; f0 < L; f0 += (int64_t)nb * F) {
    const bool act = e < nf && f0 + fl < L;
    const int64_t idx = f0 + fl + L * e;
    if (act) Xs[t] = __ldcg(&a.T2[idx]);
    __syncthreads();
    double s = 0.0;
    if (act) {
      for (int k = c; k < r3; ++k) s = fma(R3[c + LD * k], Xs[fl + F * (k + r3 * dd)], s);
      if (d.p == 4) Ys[t] = s;
    }
    __syncthreads();
    if (act) {
      if (d.p == 4) {
        s = 0.0;
        for (int k = dd; k < r4; ++k) s = fma(R4[dd + LD * k], Ys[fl + F * (c + r3 * k)], s);
      }
      a.T[idx] = s;
      if (sizeof(Tc) == 4) ((float*)a.Tcore)[idx] = (float)s;
    }
  }
}

// The row tiles of all modes, numbered mode after mode.
struct RowTiles {
  int base[kMaxModes + 1];
  bool tree;                               // a mode above kTreeTiles row tiles
  __device__ explicit RowTiles(const ModeDesc& d) {
    int tot = 0;
    tree = false;
    for (int n = 0; n < d.p; ++n) {
      const int nt = (int)((d.N[n] + 31) / 32);
      base[n] = tot;
      tot += nt;
      tree |= nt > kTreeTiles;
    }
    for (int n = d.p; n <= kMaxModes; ++n) base[n] = tot;
  }
  __device__ int total() const { return base[kMaxModes]; }
  __device__ void find(int task, int* n_out, int* t_out) const {
    int n = 0;
    while (task >= base[n + 1]) ++n;
    *n_out = n;
    *t_out = task - base[n];
  }
};

// Phase 1: M, X, partial P; dS = Y_2 x_2 A_2^T when the projection left it.  (Every phase takes
// the CTA's index among the nb that share the state: the whole grid, or a member's part of a
// batch's.  The values do not depend on nb.)
template <typename Tc>
__device__ void phase_rows1(const UpdArgs& a, const RowTiles& rt, unsigned char* smraw, unsigned bid, unsigned nb) {
  const ModeDesc& d = a.d;
  for (int task = bid; task < rt.total(); task += nb) {
    int n, t;
    rt.find(task, &n, &t);
    rows_mxp<Tc>(a, n, (int64_t)t * 32, t, smraw);
  }
  // (dS on the CTAs without rows where those hold all of it at once, else on all)
  const unsigned dsc0 = (int64_t)nb - rt.total() >= update_ds_ctas(prod_r(d)) ? (unsigned)rt.total() : 0u;
  if (!a.ds_y2 || bid < dsc0) return;
  // dS = Y_2 x_2 A_2^T (Eqs. 2.15/2.16: dS = Y_n x_n A_n^T for every n), read from phase 4 on.
  // Eight consecutive threads share one element: each sums every eighth i2 with all its loads
  // in flight, then the eight partial sums are added by shuffles in a fixed order.
  const Tc* Y2 = (const Tc*)a.ds_y2;
  const Tc* A2 = (const Tc*)a.A[1];
  const int r1 = d.r[0], r2 = d.r[1];
  const int N2 = (int)d.N[1];
  const int64_t tot = prod_r(d);
  const int grp = threadIdx.x >> 3, part = threadIdx.x & 7;
  const int ngrp = blockDim.x >> 3;
  const int64_t stride = (int64_t)(nb - dsc0) * ngrp;
  const int64_t rounds = (tot + stride - 1) / stride;
  for (int64_t k = 0; k < rounds; ++k) {
    const int64_t e = (bid - dsc0) + (int64_t)(nb - dsc0) * grp + stride * k;
    Tc acc = Tc(0);
    if (e < tot) {
      const int a1 = (int)(e % r1);
      const int64_t rest = e / r1;
      const int b = (int)(rest % r2);
      const int64_t q = rest / r2;
      const Tc* y = Y2 + a1 + (int64_t)r1 * N2 * q;      // Y_2[a1 + r1 (i2 + N2 q)]
      const Tc* A = A2 + (int64_t)N2 * b;
#pragma unroll 16
      for (int i2 = part; i2 < N2; i2 += 8) acc += __ldcg(&y[(int64_t)r1 * i2]) * A[i2];
    }
    acc += __shfl_xor_sync(0xffffffffu, acc, 4);
    acc += __shfl_xor_sync(0xffffffffu, acc, 2);
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    if (e < tot && part == 0) ((Tc*)a.dS_out)[e] = acc;
  }
}

// Phase 2: P, U', partial C
template <typename Tc>
__device__ void phase_rows2(const UpdArgs& a, const RowTiles& rt, unsigned char* smraw, unsigned bid, unsigned nb) {
  for (int task = bid; task < rt.total(); task += nb) {
    int n, t;
    rt.find(task, &n, &t);
    rows_u1<Tc>(a, n, (int64_t)t * 32, t, smraw);
  }
}

// Phase 3: Cholesky-QR factors of the mode of this CTA's rows; U''
template <typename Tc>
__device__ void phase_rows3(const UpdArgs& a, const RowTiles& rt, unsigned char* smraw, unsigned bid, unsigned nb) {
  double* Rs = (double*)smraw;
  int have = -1;
  for (int task = bid; task < rt.total(); task += nb) {
    int n, t;
    rt.find(task, &n, &t);
    if (n != have) mode_cholqr<Tc>(a, n, smraw, t == 0);
    have = n;
    rows_u2<Tc>(a, n, (int64_t)t * 32, Rs + LD * LD, (unsigned char*)(Rs + 2 * LD * LD));
    if (t == 0) {
      a.R[(int64_t)n * LD * LD + threadIdx.x] = Rs[threadIdx.x];
      a.Rinv[(int64_t)n * LD * LD + threadIdx.x] = Rs[LD * LD + threadIdx.x];
    }
  }
}

// Phase 6: Gram partials
template <typename Tc>
__device__ void phase_grams(const UpdArgs& a, unsigned char* smraw, unsigned bid, unsigned nb) {
  for (int task = bid; task < a.d.p * a.gsplit; task += nb)
    gram_partial<sizeof(Tc) == 4 ? 4 : 1>(a.d, a.T, a.gpart, a.gsplit, task / a.gsplit, task % a.gsplit,
                                          (double(*)[33])smraw);
}

template <typename Tc>
__global__ void __launch_bounds__(UPD_THREADS, 1) k_update(UpdArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int abort_sh;
  if (threadIdx.x == 0) abort_sh = 0;
  __syncthreads();
  __shared__ unsigned long long st_sh[16];
  int nst = 0;                             // kUpdPhases at the end, whatever p
  unsigned nbar = 0;
  stamp(st_sh, a.stamps, 0);
  const int p = a.d.p;
  const unsigned bid = blockIdx.x, nb = gridDim.x;
  const RowTiles rt(a.d);
  phase_rows1<Tc>(a, rt, smraw, bid, nb);
  if (!grid_sync(a.bar, ++nbar, nb, a.flags, &abort_sh)) return;
  stamp(st_sh, a.stamps, ++nst);
  if (rt.tree) {
    reduce_long<Tc>(a, 0, bid, nb);
    if (!grid_sync(a.bar, ++nbar, nb, a.flags, &abort_sh)) return;
  }
  phase_rows2<Tc>(a, rt, smraw, bid, nb);
  if (!grid_sync(a.bar, ++nbar, nb, a.flags, &abort_sh)) return;
  stamp(st_sh, a.stamps, ++nst);
  if (rt.tree && a.reorth) {
    reduce_long<Tc>(a, 1, bid, nb);
    if (!grid_sync(a.bar, ++nbar, nb, a.flags, &abort_sh)) return;
  }
  phase_rows3<Tc>(a, rt, smraw, bid, nb);
  if (!grid_sync(a.bar, ++nbar, nb, a.flags, &abort_sh)) return;
  stamp(st_sh, a.stamps, ++nst);
  core_12<Tc>(a, smraw, bid, nb);
  if (!grid_sync(a.bar, ++nbar, nb, a.flags, &abort_sh)) return;
  stamp(st_sh, a.stamps, ++nst);
  if (p > 2) {
    core_34<Tc>(a, smraw, bid, nb);
    if (!grid_sync(a.bar, ++nbar, nb, a.flags, &abort_sh)) return;
  }
  stamp(st_sh, a.stamps, ++nst);
  phase_grams<Tc>(a, smraw, bid, nb);
  if (a.skip_finish) {
    // (the finish is another launch: the kernel's end orders it)
    stamp(st_sh, a.stamps, ++nst);
    stamp(st_sh, a.stamps, ++nst);
    stamp_flush(st_sh, a.stamps, nst);
    return;
  }
  if (!grid_sync(a.bar, ++nbar, nb, a.flags, &abort_sh)) return;
  stamp(st_sh, a.stamps, ++nst);
  // 7: G, G^{-1}, sigma^2 (or a separate launch beside the exact error)
  for (int n = bid; n < p; n += nb)
    gram_finish(a.d, n, a.gpart, a.gsplit, a.G, a.Ginv, a.Ginvf, a.sig2, a.Vprev, a.warm, a.flags, smraw);
  stamp(st_sh, a.stamps, ++nst);
  stamp_flush(st_sh, a.stamps, nst);
}

// One phase of the updates of up to kUpdBatch states (members of a batch) in an ordinary
// launch: CTAs base[m] .. base[m + 1] - 1 are member m's.  The phases are the fused kernel's,
// the end of a launch taking the place of the grid barrier, so that no member's CTAs hold an
// SM while they wait and none needs to be resident with the others of its grid.
struct UpdBatch {
  int n;
  int base[kUpdBatch + 1];
  UpdArgs a[kUpdBatch];
};
enum { PH_ROWS1, PH_SUM_P, PH_ROWS2, PH_SUM_C, PH_ROWS3, PH_CORE12, PH_CORE34, PH_GRAMS, PH_FINISH };
template <typename Tc, int PH>
__global__ void __launch_bounds__(UPD_THREADS, 1) k_update_batch(const __grid_constant__ UpdBatch B) {
  extern __shared__ __align__(16) unsigned char smraw[];
  int m = 0;
  while ((int)blockIdx.x >= B.base[m + 1]) ++m;
  const UpdArgs& a = B.a[m];
  const unsigned bid = blockIdx.x - B.base[m], nb = B.base[m + 1] - B.base[m];
  if constexpr (PH == PH_CORE12) {
    core_12<Tc>(a, smraw, bid, nb);
  } else if constexpr (PH == PH_CORE34) {
    core_34<Tc>(a, smraw, bid, nb);
  } else if constexpr (PH == PH_GRAMS) {
    phase_grams<Tc>(a, smraw, bid, nb);
  } else if constexpr (PH == PH_FINISH) {
    gram_finish(a.d, bid, a.gpart, a.gsplit, a.G, a.Ginv, a.Ginvf, a.sig2, a.Vprev, a.warm, a.flags, smraw);
  } else if constexpr (PH == PH_SUM_P || PH == PH_SUM_C) {
    reduce_long<Tc>(a, PH == PH_SUM_C, bid, nb);
  } else {
    const RowTiles rt(a.d);
    if constexpr (PH == PH_ROWS1) phase_rows1<Tc>(a, rt, smraw, bid, nb);
    else if constexpr (PH == PH_ROWS2) phase_rows2<Tc>(a, rt, smraw, bid, nb);
    else phase_rows3<Tc>(a, rt, smraw, bid, nb);
  }
}

// The Gram refresh of phases 6-7 as two ordinary launches (after (re)initialisation
// and state loads), bit-identical to the fused path of the same compute type.
template <int CH>
__global__ void __launch_bounds__(UPD_THREADS, 1) k_gram_partial(ModeDesc d, const double* T, double* gpart,
                                                                 int gsplit) {
  __shared__ double S[32][33];
  gram_partial<CH>(d, T, gpart, gsplit, blockIdx.x / gsplit, blockIdx.x % gsplit, S);
}

__global__ void __launch_bounds__(UPD_THREADS, 1) k_gram_finish(ModeDesc d, const double* gpart, int gsplit, double* G,
                                                                double* Ginv, float* Ginvf, double* sig2,
                                                                float* Vprev, int warm, unsigned* flags) {
  extern __shared__ __align__(16) unsigned char smraw[];
  gram_finish(d, blockIdx.x, gpart, gsplit, G, Ginv, Ginvf, sig2, Vprev, warm, flags, smraw);
}

void launch_gram_finish(const ModeDesc& d, const double* Gpart, int nsplit, double* G, double* Ginv, float* Ginvf,
                        double* sig2, float* Vprev, int warm, unsigned* flags, cudaStream_t s) {
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_gram_finish, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kUpdSmem);
    attr = true;
  }
  k_gram_finish<<<d.p, UPD_THREADS, kUpdSmem, s>>>(d, Gpart, nsplit, G, Ginv, Ginvf, sig2, Vprev, warm, flags);
  count_launch();
}

void launch_gram(const ModeDesc& d, const double* T, double* Gpart, int nsplit, double* G, double* Ginv,
                 float* Ginvf, double* sig2, float* Vprev, int warm, unsigned* flags, cudaStream_t s) {
  if (Ginvf) k_gram_partial<4><<<d.p * nsplit, UPD_THREADS, 0, s>>>(d, T, Gpart, nsplit);
  else k_gram_partial<1><<<d.p * nsplit, UPD_THREADS, 0, s>>>(d, T, Gpart, nsplit);
  count_launch();
  launch_gram_finish(d, Gpart, nsplit, G, Ginv, Ginvf, sig2, Vprev, warm, flags, s);
}

template <typename Tc>
tdb_status launch_update(UpdArgs& a, int grid_hint, cudaStream_t s) {
  static int nsm_cache[2] = {0, 0};
  int& nsm = nsm_cache[sizeof(Tc) == 8 ? 1 : 0];
  if (nsm == 0) {
    int dev = 0, n = 0, coop = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (!coop) return TDB_ERR_UNSUPPORTED;
    cudaFuncSetAttribute(k_update<Tc>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kUpdSmem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_update<Tc>, UPD_THREADS, kUpdSmem);
    if (per_sm < 1) return TDB_ERR_UNSUPPORTED;
    nsm = n;
  }
  // every CTA is resident (one per SM at most), so the grid barriers cannot deadlock
  const int grid = std::max(a.d.p, std::min(nsm, grid_hint));
  // cooperative launch through the extensible API, which stream capture records as a
  // cooperative kernel node
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(UPD_THREADS);
  cfg.dynamicSmemBytes = kUpdSmem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, k_update<Tc>, a);
  count_launch();
  return e == cudaSuccess ? TDB_OK : TDB_ERR_CUDA;
}
template tdb_status launch_update<float>(UpdArgs&, int, cudaStream_t);
template tdb_status launch_update<double>(UpdArgs&, int, cudaStream_t);

namespace {
template <int PH>
void launch_phase(UpdBatch& B, cudaStream_t s) {
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_update_batch<float, PH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kUpdSmem);
    attr = true;
  }
  if (B.base[B.n] == 0) return;
  k_update_batch<float, PH><<<B.base[B.n], UPD_THREADS, kUpdSmem, s>>>(B);
  count_launch();
}
}  // namespace

void launch_update_batch(const UpdArgs* args, int n, int part, cudaStream_t s) {
  for (int i0 = 0; i0 < n; i0 += kUpdBatch) {
    UpdBatch B;
    B.n = std::min(kUpdBatch, n - i0);
    bool tree = false, tree_c = false;
    for (int m = 0; m < B.n; ++m) {
      B.a[m] = args[i0 + m];
      for (int k = 0; k < B.a[m].d.p; ++k)
        if ((B.a[m].d.N[k] + 31) / 32 > kTreeTiles) {
          tree = true;
          tree_c |= B.a[m].reorth != 0;
        }
    }
    // a phase's CTAs per member
    auto count = [&](auto&& of) {
      B.base[0] = 0;
      for (int m = 0; m < B.n; ++m) B.base[m + 1] = B.base[m] + (int)std::min<int64_t>(of(B.a[m]), 1 << 16);
    };
    auto tiles = [](const UpdArgs& a) {
      int64_t t = 0;
      for (int k = 0; k < a.d.p; ++k) t += (a.d.N[k] + 31) / 32;
      return t;
    };
    if (part == 1) {
      count([](const UpdArgs& a) { return (int64_t)a.d.p; });
      launch_phase<PH_FINISH>(B, s);
      continue;
    }
    count([&](const UpdArgs& a) { return tiles(a) + (a.ds_y2 ? std::min<int64_t>(update_ds_ctas(prod_r(a.d)), 16) : 0); });
    launch_phase<PH_ROWS1>(B, s);
    if (tree) {
      count([](const UpdArgs& a) { return (int64_t)a.d.p * 8; });
      launch_phase<PH_SUM_P>(B, s);
    }
    count(tiles);
    launch_phase<PH_ROWS2>(B, s);
    if (tree_c) {
      count([](const UpdArgs& a) { return a.reorth ? (int64_t)a.d.p * 8 : (int64_t)0; });
      launch_phase<PH_SUM_C>(B, s);
    }
    count(tiles);
    launch_phase<PH_ROWS3>(B, s);
    count([](const UpdArgs& a) { return std::min<int64_t>(prod_r_above(a.d, 1), 16); });
    launch_phase<PH_CORE12>(B, s);
    count([](const UpdArgs& a) { return a.d.p > 2 ? std::min<int64_t>((prod_r(a.d) + 1023) / 1024, 16) : (int64_t)0; });
    launch_phase<PH_CORE34>(B, s);
    count([](const UpdArgs& a) { return (int64_t)a.d.p * a.gsplit; });
    launch_phase<PH_GRAMS>(B, s);
  }
}

// ---------------------------------------------------------------------------
// Diagnostics (tdb_selftest_recip, tdb_selftest_timeout): the double reciprocal helpers
// over an array, and the update kernel's grid barrier waiting for one CTA more than the
// grid holds - an arrival that never comes - so that its bounded wait runs out.
// ---------------------------------------------------------------------------
__global__ void k_selftest_recip(const double* __restrict__ x, double* __restrict__ rcp, double* __restrict__ rs,
                                 int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double v = x[i];
    rcp[i] = drcp(v);
    rs[i] = v > 0.0 ? drsqrt(v) : 0.0;
  }
}

__global__ void k_selftest_gridwait(unsigned* bar, unsigned* flags, long long limit) {
  __shared__ int abort_sh;
  if (threadIdx.x == 0) abort_sh = 0;
  grid_sync(bar, 1u, gridDim.x + 1u, flags, &abort_sh, limit);
}

}  // namespace tdb

extern "C" tdb_status tdb_selftest_recip(const double* x, double* rcp, double* rsqrt, int64_t n, void* stream) {
  using namespace tdb;
  if (!x || !rcp || !rsqrt || n < 0) return TDB_ERR_INVALID_ARG;
  if (n == 0) return TDB_OK;
  cudaStream_t s = (cudaStream_t)stream;
  const int blocks = (int)std::min<int64_t>((n + 255) / 256, 1024);
  k_selftest_recip<<<blocks, 256, 0, s>>>(x, rcp, rsqrt, n);
  count_launch();
  if (cudaGetLastError() != cudaSuccess) return TDB_ERR_CUDA;
  return cudaStreamSynchronize(s) == cudaSuccess ? TDB_OK : TDB_ERR_CUDA;
}

extern "C" tdb_status tdb_selftest_timeout(int which, int64_t limit_cycles, unsigned* scratch, void* stream) {
  using namespace tdb;
  if (!scratch || limit_cycles < 1 || limit_cycles > 4000000000ll || (which != 0 && which != 1))
    return TDB_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaMemsetAsync(scratch, 0, 4 * sizeof(unsigned), s) != cudaSuccess) return TDB_ERR_CUDA;
  unsigned* flags = scratch + 2;
  if (which == 0) {
    // two co-resident CTAs (cooperative launch): the barrier's target is three arrivals
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2);
    cfg.blockDim = dim3(32);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, k_selftest_gridwait, scratch, flags, (long long)limit_cycles) != cudaSuccess)
      return TDB_ERR_CUDA;
    count_launch();
  } else {
    const tdb_status st = tc_selftest_mbar_wait(flags, (long long)limit_cycles, s);
    if (st != TDB_OK) return st;
  }
  unsigned h = 0;
  if (cudaMemcpyAsync(&h, flags, sizeof(unsigned), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return TDB_ERR_CUDA;
  return (h & kFlagTimeout) ? TDB_ERR_TIMEOUT : TDB_OK;
}
