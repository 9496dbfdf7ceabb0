// proj_finish.cuh - the finishing launches of a projection pass (Eqs. 2.15/2.16): from the
// per-tile partial first contractions Z1 and Z2 that a projection kernel leaves (tc_project.cu
// on the tensor cores, simt_project.cu in float and double) to every Y_n, and ||dV||_W^2.
#pragma once
#include <cstring>

#include "kernels.h"

namespace tdb {
namespace {

__device__ __forceinline__ void fin_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void fin_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Finish, first launch.  A projection kernel leaves partial first contractions over the
// tiles q of the contracted mode: Z1p at e + n1 (s + S q), e = i2 + N2 a, n1 = r1 N2
// (mode 1 contracted), and Z2p at f + n2 (s + S q), f = i1 + N1 b, n2 = N1 r2 (mode 2
// contracted), s the slice (i3 + N3 i4).  This launch sums them over q and contracts the
// slices with B (S x J):
//   Y_2[a + r1 (i2 + N2 j)] = sum_s Z1[e, s] B[s, j],    Y_1[f + n2 j] = sum_s Z2[f, s] B[s, j],
// with B = A_3 (three modes), B[i3 + N3 i4, c + r3 d] = A_3[i3, c] A_4[i4, d] (four modes,
// the Kronecker product that contracts modes 3 and 4 at once) or the 1 x 1 identity (two
// modes).  It also writes Z1 = sum_q Z1p when there is more than one tile along mode 1
// (the next launch forms Y_3 from it) and, in its first CTA, ||dV||_W^2 from the fused
// kernel's per-CTA partials.  A CTA owns 256 elements of one side (a thread per element,
// its slice values in registers) and one of `nsplit` slice ranges; the slices' rows of B
// are staged in shared memory and read as float4 broadcasts, 32 outputs j at a time.
// With nsplit > 1 each CTA writes its partial and k_finish_red adds the partials of
// every output in split order (so results do not vary from run to run).
constexpr int FS_TE = 256, FS_SC = 16, FS_JMAX = 128, FS_SPLIT_MAX = 32;
constexpr int FS_CTAS = 2 * 152;   // split target: about two CTAs per SM
constexpr int FS_NQ_MAX = 8;   // tiles along mode 1 or 2 loaded at once; more are added in order after them
template <typename T>
struct FinArgs {
  const T* Z1p;
  const T* Z2p;
  int N1, N2, S, nq1, nq2, r1, r2;
  const T* A3;           // N3 x r3 (null: two modes, B = [1])
  const T* A4;           // N4 x r4 (null: three modes)
  int N3, r3, N4, r4, J;
  T* Z1;                 // N2 x r1 x S, i2 fastest (written when nq1 > 1 and W is not fused)
  // W = Z1 x_2 A_2^T (r1 x r2 x S: Y_3 for three modes) formed here when a first-side CTA
  // holds whole i2 columns (te1 = N2 floor(256 / N2) elements, N2 <= 256)
  T* W;
  const T* A2;
  int fuse_w, te1;
  T* Y2;
  T* Y1;
  T* part;               // [tile][split][J][256]
  int nsplit, nt1, nt2;
  const double* npart;
  int nnp;
  unsigned long long* span;     // profiling words of the main kernel (see Params), or null
  double* dv2;
};

// Row stride of A_2 in the fused finish's shared memory: = 4 (mod 32), so that the lanes
// of a warp (eight columns b x four i2 phases) read 32 different banks.  Never above that of
// N2 = FS_TE for the N2 up to FS_TE that it serves.
__host__ __device__ constexpr int a2_stride(int N2) { return N2 + ((36 - N2 % 32) % 32); }

// Four consecutive values in shared memory (16-byte aligned).
template <typename T>
struct __align__(16) Quad {
  T x, y, z, w;
};

// acc[0 .. 3] += b z; float as two pairs of multiply-adds (one issue slot each).
__device__ __forceinline__ void fma4(double (&acc)[4], const Quad<double>& b, double z) {
  acc[0] = fma(b.x, z, acc[0]);
  acc[1] = fma(b.y, z, acc[1]);
  acc[2] = fma(b.z, z, acc[2]);
  acc[3] = fma(b.w, z, acc[3]);
}
__device__ __forceinline__ void fma4(float (&acc)[4], const Quad<float>& b, float z) {
  const float2 zz = make_float2(z, z);
  const float2 lo = __ffma2_rn(make_float2(b.x, b.y), zz, make_float2(acc[0], acc[1]));
  const float2 hi = __ffma2_rn(make_float2(b.z, b.w), zz, make_float2(acc[2], acc[3]));
  acc[0] = lo.x;
  acc[1] = lo.y;
  acc[2] = hi.x;
  acc[3] = hi.y;
}

// W[a1, b, s] = sum_i2 Z1[i2, a1, s] A2[i2, b] of a finish CTA's whole columns a1 = a1_lo + al
// (al < na) and sc staged slices: eight lanes share a tile of TU slices x 8 / TU columns b, each
// taking every eighth run of VEC values of i2 (the lanes' runs are neighbours: no bank
// conflicts), and a transposing butterfly leaves one sum to each lane.
template <typename T, int VEC, int TU>
__device__ __forceinline__ void finish_w(const FinArgs<T>& f, const T* zs, const T* a2s, int a2st, int na, int a1_lo,
                                         int s0, int sc) {
  constexpr int TB = 8 / TU;
  const int kp = threadIdx.x & 7, nbg = (f.r2 + TB - 1) / TB, nug = (sc + TU - 1) / TU;
  const int ntile = nbg * nug * na;
  for (int t0 = 4 * (threadIdx.x >> 5); t0 < ntile; t0 += FS_TE / 8) {      // four tiles a warp
    const int mine = t0 + ((threadIdx.x >> 3) & 3), tile = min(mine, ntile - 1);
    const int bg = tile % nbg, rest = tile / nbg, ug = rest % nug, al = rest / nug;
    const T* zc = zs + TU * ug * FS_TE + al * f.N2;
    T w[8];                                                // [b][u]
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = T(0);
    for (int i2 = VEC * kp; i2 < f.N2; i2 += 8 * VEC) {
      if constexpr (VEC == 4) {
        Quad<T> z[TU];
#pragma unroll
        for (int u = 0; u < TU; ++u) z[u] = *reinterpret_cast<const Quad<T>*>(zc + u * FS_TE + i2);
#pragma unroll
        for (int b = 0; b < TB; ++b) {
          const Quad<T> x = *reinterpret_cast<const Quad<T>*>(a2s + a2st * min(TB * bg + b, f.r2 - 1) + i2);
#pragma unroll
          for (int u = 0; u < TU; ++u)
            w[TU * b + u] = fma(z[u].x, x.x, fma(z[u].y, x.y, fma(z[u].z, x.z, fma(z[u].w, x.w, w[TU * b + u]))));
        }
      } else {
        T z[TU];
#pragma unroll
        for (int u = 0; u < TU; ++u) z[u] = zc[u * FS_TE + i2];
#pragma unroll
        for (int b = 0; b < TB; ++b) {
          const T x = a2s[a2st * min(TB * bg + b, f.r2 - 1) + i2];
#pragma unroll
          for (int u = 0; u < TU; ++u) w[TU * b + u] = fma(z[u], x, w[TU * b + u]);
        }
      }
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      const bool up = kp & o;
#pragma unroll
      for (int i = 0; i < o; ++i) {
        const T keep = up ? w[i + o] : w[i], send = up ? w[i] : w[i + o];
        w[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
    }
    const int u = TU * ug + kp % TU, b = TB * bg + kp / TU, a = a1_lo + al;
    if (mine < ntile && u < sc && b < f.r2 && a < f.r1)
      f.W[a + (int64_t)f.r1 * (b + (int64_t)f.r2 * (s0 + u))] = w[0];
  }
}

// NQ: tiles along the contracted mode, rounded up to a power of two (<= FS_NQ_MAX); JB:
// outputs j at a time (float 8, 16, 32 or 64, the least that holds all J, with fewer slices at
// 64; double 8, and half of the slices: two CTAs per SM within 128 registers a thread).
// Bound: latency of the partials, chunk after chunk.  256 x 128 x 512 at ranks (11, 8, 16) 13.6
// us cold (19.9 with 32 outputs tested in groups of four, chunks of 16 and 7 slices and a
// thread per W output), 192 x 129 x 192 x 3 at (13, 3, 15, 3), 45 outputs, 22 us (27: the partials read
// once per 32 outputs), 126^3 double 31.8 us (33.2).
template <typename T, int NQ, int JB>
__global__ void __launch_bounds__(FS_TE, 2) k_finish_sk(FinArgs<T> f) {
  constexpr int WIDE = sizeof(T) / 4;                                       // 1 float, 2 double
  constexpr int SC0 = (NQ <= 2 ? FS_SC : (NQ == 4 ? FS_SC / 2 : FS_SC / 4)) / WIDE;
  constexpr int SC = JB == 64 && SC0 > FS_SC / 2 ? FS_SC / 2 : SC0;         // slices per chunk
  constexpr bool ONE = sizeof(T) == 4 && JB <= 32;          // J <= JB: one pass over j
  constexpr int BPT = (SC * (ONE ? JB : FS_JMAX) + FS_TE - 1) / FS_TE;   // B values a thread stages per chunk
  extern __shared__ __align__(16) unsigned char fs_raw[];
  T* fs_sm = (T*)fs_raw;                            // B rows of a slice chunk: [FS_SC][Jp]
  __shared__ double dsh[32];
  const int tid = threadIdx.x;
  if (tid == 0) fin_dep_launch();
  const int tile = blockIdx.x / f.nsplit, sp = blockIdx.x % f.nsplit;
  const bool first = tile < f.nt1;
  const bool fw = first && f.fuse_w;
  const int Jp0 = (f.J + 3) & ~3;
  T* zs = fs_sm + FS_SC * Jp0;                         // fw: the chunk's z values [FS_SC][FS_TE]
  T* a2s = zs + FS_SC * FS_TE;                     // fw: A_2 (N2 x r2, ld a2_stride(N2))
  const int a2st = a2_stride(f.N2);
  if (fw) {
    // A_2 is an input of the step (not written by the main kernel): staged before the wait
    for (int i0 = tid; i0 < f.N2 * f.r2; i0 += 4 * FS_TE) {
      T v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = i0 + k * FS_TE < f.N2 * f.r2 ? __ldg(&f.A2[i0 + k * FS_TE]) : T(0);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int idx = i0 + k * FS_TE;
        if (idx < f.N2 * f.r2) a2s[idx % f.N2 + a2st * (idx / f.N2)] = v[k];
      }
    }
  }
  // programmatic launch: the main kernel's results (partials, norms, span words) are
  // complete and visible after this
  fin_dep_wait();
  if (blockIdx.x == gridDim.x - 1) {
    // ||dV||_W^2: the main kernel's partials, eight loads in flight per thread (in the last
    // CTA, a second-side one whenever there is one: those form no W)
    double t = 0.0;
    for (int i0 = tid; i0 < f.nnp; i0 += 8 * FS_TE) {
      double v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = i0 + k * FS_TE < f.nnp ? __ldcg(&f.npart[i0 + k * FS_TE]) : 0.0;
#pragma unroll
      for (int k = 0; k < 8; ++k) t += v[k];
    }
    t = block_sum(t, dsh);
    if (tid == 0) *f.dv2 = t;
    if (tid == 0 && f.span) {
      // the main kernel has completed: its span into the sums, the words reset for the next
      const unsigned long long a = f.span[0], b = f.span[1];
      if (b > a) {
        f.span[2] += b - a;
        f.span[3] += 1;
      }
      f.span[0] = ~0ull;
      f.span[1] = 0ull;
    }
  }
  const int64_t ne = first ? (int64_t)f.r1 * f.N2 : (int64_t)f.N1 * f.r2;
  const int te = first ? f.te1 : FS_TE;                // elements per CTA on this side
  const int64_t e = (int64_t)(first ? tile : tile - f.nt1) * te + tid;
  const bool in = tid < te && e < ne;
  const int na = fw ? te / f.N2 : 0;                   // a1 values this CTA holds whole
  const int a1_lo = fw ? tile * na : 0;
  const int nq = first ? f.nq1 : f.nq2;
  const T* Pp = (first ? f.Z1p : f.Z2p) + (in ? e : 0);
  const bool write_z = first && f.nq1 > 1 && !f.fuse_w;
  const int J = f.J, Jp = (J + 3) & ~3;
  const int s_lo = (int)((int64_t)f.S * sp / f.nsplit), s_hi = (int)((int64_t)f.S * (sp + 1) / f.nsplit);
  const int64_t qstride = ne * (int64_t)f.S;
  T* mine = f.part + ((int64_t)tile * f.nsplit + sp) * (int64_t)J * FS_TE;
  auto store = [&](int64_t ee, int j, T v) {
    if (first) {
      const int64_t a = ee / f.N2, i2 = ee - a * f.N2;
      f.Y2[a + (int64_t)f.r1 * i2 + ne * (int64_t)j] = v;
    } else {
      f.Y1[ee + ne * (int64_t)j] = v;
    }
  };
  // chunks of equal length (at most SC slices)
  const int nch = (s_hi - s_lo + SC - 1) / SC;
  for (int j0 = 0; j0 < (ONE ? 1 : J); j0 += JB) {
    const int jn = min(JB, J - j0);
    T acc[JB / 4][4];
#pragma unroll
    for (int t = 0; t < JB; ++t) acc[t / 4][t % 4] = T(0);
    for (int ch = 0; ch < nch; ++ch) {
      const int s0 = s_lo + (s_hi - s_lo) * ch / nch;
      const int sc = s_lo + (s_hi - s_lo) * (ch + 1) / nch - s0;
      // this element's slice values summed over q: every load of the chunk is issued
      // into registers before the first addition
      T raw[SC * NQ];
#pragma unroll
      for (int u = 0; u < SC; ++u) {
        const T* pe = Pp + ne * (int64_t)(s0 + u);
#pragma unroll
        for (int q = 0; q < NQ; ++q) raw[u * NQ + q] = (in && u < sc && q < nq) ? __ldcg(pe + qstride * q) : T(0);
      }
      // this chunk's B rows, loaded beside the partials (staged in shared memory below)
      T bpre[BPT];
#pragma unroll
      for (int k = 0; k < BPT; ++k) {
        const int idx = tid + k * FS_TE;
        T bv = T(0);
        if (idx < SC * Jp) {
          const int sl = idx % SC, j = idx / SC;       // consecutive threads: consecutive slices
          if (sl < sc && j < J) {
            const int s = s0 + sl;
            if (!f.A3) {
              bv = T(1);
            } else if (!f.A4) {
              bv = __ldg(&f.A3[s + (int64_t)f.N3 * j]);
            } else {
              const int i3 = s % f.N3, i4 = s / f.N3, c = j % f.r3, dd = j / f.r3;
              bv = __ldg(&f.A3[i3 + (int64_t)f.N3 * c]) * __ldg(&f.A4[i4 + (int64_t)f.N4 * dd]);
            }
          }
        }
        bpre[k] = bv;
      }
      T z[SC];
#pragma unroll
      for (int u = 0; u < SC; ++u) {
        T v = raw[u * NQ];
#pragma unroll
        for (int q = 1; q < NQ; ++q) v += raw[u * NQ + q];
        if (NQ == FS_NQ_MAX && nq > NQ && in && u < sc) {
          // a long mode (more than FS_NQ_MAX tiles): the rest in tile order
          const T* pe = Pp + ne * (int64_t)(s0 + u);
          for (int q = NQ; q < nq; ++q) v += __ldcg(pe + qstride * q);
        }
        z[u] = v;
      }
      if (write_z && j0 == 0 && in) {
#pragma unroll
        for (int u = 0; u < SC; ++u)
          if (u < sc) f.Z1[e + ne * (int64_t)(s0 + u)] = z[u];
      }
      __syncthreads();                                   // the previous chunk is done with zs, fs_sm
      if (fw && j0 == 0) {
#pragma unroll
        for (int u = 0; u < SC; ++u) zs[u * FS_TE + tid] = (in && u < sc) ? z[u] : T(0);
      }
#pragma unroll
      for (int k = 0; k < BPT; ++k) {
        const int idx = tid + k * FS_TE;
        if (idx < SC * Jp) fs_sm[(idx % SC) * Jp + idx / SC] = bpre[k];
      }
      __syncthreads();
      if (fw && j0 == 0) {
        constexpr int TU = SC < 4 ? SC : 4;
        if ((f.N2 & 3) == 0) finish_w<T, 4, TU>(f, zs, a2s, a2st, na, a1_lo, s0, sc);
        else finish_w<T, 1, TU>(f, zs, a2s, a2st, na, a1_lo, s0, sc);
      }
#pragma unroll
      for (int u = 0; u < SC; ++u) {
        if (u >= sc) break;
        const T* brow = fs_sm + u * Jp + j0;
#pragma unroll
        for (int t4 = 0; t4 < JB / 4; ++t4)
          if (4 * t4 < jn) fma4(acc[t4], *reinterpret_cast<const Quad<T>*>(brow + 4 * t4), z[u]);
      }
    }
    if (f.nsplit == 1) {
      if (in) {
#pragma unroll
        for (int t = 0; t < JB; ++t)
          if (t < jn) store(e, j0 + t, acc[t / 4][t % 4]);
      }
    } else {
#pragma unroll
      for (int t = 0; t < JB; ++t)
        if (t < jn) mine[(int64_t)(j0 + t) * FS_TE + tid] = acc[t / 4][t % 4];
    }
  }
}

// Finish, split partials: output (e, j) of a tile is the sum of its nsplit partials in
// split order (one thread per output, every load issued before the additions).
template <typename T>
__global__ void __launch_bounds__(256) k_finish_red(FinArgs<T> f) {
  fin_dep_wait();                  // programmatic launch: the split partials are complete
  const int J = f.J;
  const int64_t per_tile = (int64_t)J * FS_TE;
  const int64_t total = (int64_t)(f.nt1 + f.nt2) * per_tile;
  for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < total; o += (int64_t)gridDim.x * blockDim.x) {
    const int tile = (int)(o / per_tile);
    const int rem = (int)(o % per_tile);
    const int j = rem / FS_TE, x = rem % FS_TE;
    const bool first = tile < f.nt1;
    const int64_t ne = first ? (int64_t)f.r1 * f.N2 : (int64_t)f.N1 * f.r2;
    const int te = first ? f.te1 : FS_TE;
    const int64_t e = (int64_t)(first ? tile : tile - f.nt1) * te + x;
    if (x >= te || e >= ne) continue;
    const T* base = f.part + (int64_t)tile * f.nsplit * per_tile + (int64_t)j * FS_TE + x;
    T vals[FS_SPLIT_MAX];
#pragma unroll
    for (int q = 0; q < FS_SPLIT_MAX; ++q) vals[q] = q < f.nsplit ? __ldcg(&base[(int64_t)q * per_tile]) : T(0);
    T v = T(0);
#pragma unroll
    for (int q = 0; q < FS_SPLIT_MAX; ++q) v += vals[q];
    if (first) {
      const int64_t a = e / f.N2, i2 = e - a * f.N2;
      f.Y2[a + (int64_t)f.r1 * i2 + ne * (int64_t)j] = v;
    } else {
      f.Y1[e + ne * (int64_t)j] = v;
    }
  }
}


// Three-mode finish, second launch: Y_3 = Z1 x_2 A_2^T (r1 x r2 x S), a CTA per
// slice, i2 in chunks of FB_CH staged in shared memory (thread per output (a1, a2)).
// dS = Y_3 x_3 A_3^T follows in the update kernel.
constexpr int FB_CH = 128;
template <typename T>
__global__ void __launch_bounds__(256) k_finish_b(const T* __restrict__ Z1, int N2, int S, int r1, int r2,
                                                  const T* __restrict__ A2, T* __restrict__ Y3) {
  extern __shared__ __align__(16) unsigned char fb_raw[];
  T* zs = (T*)fb_raw;                  // r1 x FB_CH (element a + r1 il), from Z1 at i2 + N2 a + r1 N2 s
  T* as = zs + 32 * FB_CH;         // FB_CH x r2 (ld FB_CH + 1)
  const int tid = threadIdx.x;
  const int64_t n1 = (int64_t)r1 * N2;
  for (int sl = blockIdx.x; sl < S; sl += gridDim.x) {
    T acc[4] = {T(0), T(0), T(0), T(0)};
    for (int i0 = 0; i0 < N2; i0 += FB_CH) {
      const int ch = min(FB_CH, N2 - i0);
      const T* src = Z1 + i0 + n1 * sl;
#pragma unroll 4
      for (int e = tid; e < r1 * ch; e += 256) {
        const int il = e % ch, a = e / ch;
        zs[a + r1 * il] = __ldcg(&src[il + (int64_t)N2 * a]);
      }
#pragma unroll 4
      for (int e = tid; e < ch * r2; e += 256) {
        const int il = e % ch, b = e / ch;
        as[il + (FB_CH + 1) * b] = __ldg(&A2[i0 + il + (int64_t)N2 * b]);
      }
      __syncthreads();
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int o = tid + 256 * j;
        const int a1 = o % r1, a2 = o / r1;
        if (a2 < r2)
          for (int il = 0; il < ch; ++il) acc[j] = fma(as[il + (FB_CH + 1) * a2], zs[a1 + r1 * il], acc[j]);
      }
      __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int o = tid + 256 * j;
      const int a1 = o % r1, a2 = o / r1;
      if (a2 < r2) Y3[a1 + (int64_t)r1 * (a2 + (int64_t)r2 * sl)] = acc[j];
    }
  }
}

// Product of the weights of modes >= 3, per slice.
__global__ void k_slice_weights(int p, const double* w3, int N3, const double* w4, int N4, double* out) {
  int n = (p >= 3 ? N3 : 1) * (p >= 4 ? N4 : 1);
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x) {
    double v = 1.0;
    if (p >= 3) v *= w3[s % N3];
    if (p >= 4) v *= w4[s / N3];
    out[s] = v;
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
// Split partials a tuned plan keeps: (FS_CTAS + tiles) x 256 x J values bound nsplit x tiles x 256 x J
// for the split counts that the tuner tries first.
inline size_t finish_part_elems(int p, const int64_t* N, const int* cap) {
  const int jmax = p == 2 ? 1 : (p == 3 ? cap[2] : cap[2] * cap[3]);
  const int64_t ntmax = ((int64_t)cap[0] * N[1] + FS_TE - 1) / FS_TE + ((int64_t)N[0] * cap[1] + FS_TE - 1) / FS_TE;
  return (size_t)(FS_CTAS + ntmax) * FS_TE * jmax;
}
inline int finish_outputs(int p, const int* r) { return p == 2 ? 1 : (p == 3 ? r[2] : r[2] * r[3]); }

// The tiling of a finish: W inside it (its first-side CTAs hold whole i2 columns), the elements of
// a first-side CTA, the tiles of both sides.
struct FinTiles {
  bool fuse_w;
  int te1, nt1, nt2;
};
inline FinTiles finish_tiles(int p, const int64_t* N, const int* r) {
  FinTiles t;
  t.fuse_w = p >= 3 && N[1] <= FS_TE;
  t.te1 = t.fuse_w ? (int)N[1] * (FS_TE / (int)N[1]) : FS_TE;
  t.nt1 = (int)((r[0] * N[1] + t.te1 - 1) / t.te1);
  t.nt2 = (int)((N[0] * r[1] + FS_TE - 1) / FS_TE);
  return t;
}
// A split takes at least 16 slices in float and 4 in double, whose arithmetic (64 cycles per
// warp instruction and sub-partition) is worth more SMs than the split's partials cost.
template <typename T>
constexpr int kFinMinSlices = sizeof(T) == 4 ? FS_SC : 4;
// Split partials (values) of the launches that aim at FS_CTAS CTAs, at any ranks up to `cap`: none
// where the slices do not split, else at most FS_CTAS tiles (or all the splits' tiles) of at most
// FS_JMAX outputs.
template <typename T>
size_t finish_split_elems(int p, const int64_t* N, const int* cap) {
  int64_t ns = 1;
  for (int n = 2; n < p; ++n) ns *= N[n];
  const int64_t most = std::min<int64_t>(FS_SPLIT_MAX, ns / kFinMinSlices<T>);
  if (most < 2) return 0;
  const FinTiles t = finish_tiles(p, N, cap);
  return (size_t)std::min<int64_t>(FS_CTAS, most * (t.nt1 + t.nt2)) * FS_TE * std::min(finish_outputs(p, cap), FS_JMAX);
}

// The finish of one projection: Y_1, Y_2 (and Z1) from the tile partials, the slices
// contracted with B = A_3 (x A_4); then Y_3 (three modes) or W = Z1 x_2 A_2^T (four modes).
// More than FS_JMAX outputs per slice (r_3 r_4 of four modes) are not taken.
template <typename T>
struct Finish {
  FinArgs<T> f;
  int p = 0, nt1 = 0, nt2 = 0, J = 0, nslice = 1, nqm = 1;
  bool fuse_w = false;
  size_t smem = 0, part_cap = 0;
  T* scratch = nullptr;          // W of four modes
  const T* z1p = nullptr;
  cudaStream_t s = nullptr;

  void setup(int p_, const int64_t* N, const int* r, const void* const* A, T* z1, const T* z1p_, const T* z2p, int nq1,
             int nq2, T* scratch_, T* const* Y, T* part, size_t part_cap_, const double* npart, double* dv2,
             cudaStream_t s_) {
    p = p_;
    s = s_;
    scratch = scratch_;
    z1p = z1p_;
    part_cap = part_cap_;
    const int N1 = (int)N[0], N2 = (int)N[1];
    nslice = 1;
    for (int n = 2; n < p; ++n) nslice *= (int)N[n];
    J = finish_outputs(p, r);
    const FinTiles t = finish_tiles(p, N, r);
    fuse_w = t.fuse_w;
    const int te1 = t.te1;
    nt1 = t.nt1;
    nt2 = t.nt2;
    nqm = std::max(nq1, nq2);
    memset(&f, 0, sizeof(f));
    f.Z1p = z1p;
    f.Z2p = z2p;
    f.N1 = N1;
    f.N2 = N2;
    f.S = nslice;
    f.nq1 = nq1;
    f.nq2 = nq2;
    f.r1 = r[0];
    f.r2 = r[1];
    f.A3 = p >= 3 ? (const T*)A[2] : nullptr;
    f.A4 = p >= 4 ? (const T*)A[3] : nullptr;
    f.N3 = p >= 3 ? (int)N[2] : 1;
    f.r3 = p >= 3 ? r[2] : 1;
    f.N4 = p >= 4 ? (int)N[3] : 1;
    f.r4 = p >= 4 ? r[3] : 1;
    f.J = J;
    f.Z1 = z1;
    f.W = p == 3 ? Y[2] : scratch;
    f.A2 = (const T*)A[1];
    f.fuse_w = fuse_w ? 1 : 0;
    f.te1 = te1;
    f.Y2 = Y[1];
    f.Y1 = Y[0];
    f.part = part;
    f.nt1 = nt1;
    f.nt2 = nt2;
    f.npart = npart;
    f.dv2 = dv2;
    smem = sizeof(T) * (FS_SC * ((J + 3) & ~3) + (fuse_w ? FS_SC * FS_TE + (size_t)a2_stride(N2) * r[1] : 0));
  }

  // splits per tile: the grid stays within the target (whole waves of resident CTAs: two
  // per SM), at least one split
  int nsplit_for(int target) const {
    int ns = (int)std::max<int64_t>(1, target / (nt1 + nt2));
    ns = std::min({ns, std::max(1, nslice / kFinMinSlices<T>), FS_SPLIT_MAX});
    while (ns > 1 && (size_t)ns * (nt1 + nt2) * FS_TE * J > part_cap) --ns;
    return ns;
  }

  // both finishing kernels start by programmatic launch behind the kernel before them (their
  // set-up overlaps its tail; they wait for it before reading its results)
  template <typename K>
  void launch_pdl(K kern, int grid, size_t sm) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(FS_TE);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kern, f);
    count_launch();
  }

  // The limit is set once, to the most that any launch needs (FS_JMAX outputs, A_2 of 32 ranks):
  // with each launch's own need another thread's smaller one could lower it just before this
  // launch, and a need of 48 KB less the static part and more was left at the default.
  static constexpr size_t smem_max = sizeof(T) * (FS_SC * FS_JMAX + FS_SC * FS_TE + (size_t)a2_stride(FS_TE) * kMaxRank);
  template <int NQ, int JB>
  void launch_sk_nq(int grid) {
    static const cudaError_t once = cudaFuncSetAttribute(
        k_finish_sk<T, NQ, JB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max);
    (void)once;
    launch_pdl(k_finish_sk<T, NQ, JB>, grid, smem);
  }
  template <int JB>
  void launch_sk(int grid) {
    if (nqm <= 1) launch_sk_nq<1, JB>(grid);
    else if (nqm <= 2) launch_sk_nq<2, JB>(grid);
    else if (nqm <= 4) launch_sk_nq<4, JB>(grid);
    else launch_sk_nq<8, JB>(grid);
  }

  void launch(int nsplit) {
    f.nsplit = nsplit;
    const int grid = (nt1 + nt2) * nsplit;
    if constexpr (sizeof(T) == 4) {
      if (J <= 8) launch_sk<8>(grid);
      else if (J <= 16) launch_sk<16>(grid);
      else if (J <= 32) launch_sk<32>(grid);
      else launch_sk<64>(grid);
    } else {
      launch_sk<8>(grid);
    }
    if (nsplit > 1) {
      const int64_t outs = (int64_t)(nt1 + nt2) * J * FS_TE;
      launch_pdl(k_finish_red<T>, (int)std::min<int64_t>((outs + 255) / 256, 152 * 16), 0);
    }
  }

  // Y_3 and Y_4 once the partials are contracted
  void launch_rest(const int64_t* N, const int* r, const void* const* A, T* const* Y) {
    if (p < 3) return;
    if (!fuse_w) {
      // Z1 summed over the mode-1 tiles: the partials themselves when there is one tile
      const T* z1 = f.nq1 > 1 ? f.Z1 : z1p;
      constexpr size_t sm = (size_t)(32 * FB_CH + 32 * (FB_CH + 1)) * sizeof(T);
      static bool attr = false;
      if (sm > 48 * 1024 && !attr) {
        cudaFuncSetAttribute(k_finish_b<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        attr = true;
      }
      k_finish_b<T><<<std::min(nslice, 152 * 8), 256, sm, s>>>(z1, f.N2, nslice, r[0], r[1], (const T*)A[1], f.W);
      count_launch();
    }
    if (p == 4) {
      // Y_3 = W x_4 A_4^T and Y_4 = W x_3 A_3^T from W = Z1 x_2 A_2^T (r1 x r2 x N3 x N4)
      const int64_t L12 = (int64_t)r[0] * r[1];
      launch_modeprod<T, T, T>(scratch, Y[2], (const T*)A[3], L12 * N[2], (int)N[3], r[3], 1, N[3], 1, s);
      launch_modeprod<T, T, T>(scratch, Y[3], (const T*)A[2], L12, (int)N[2], r[2], N[3], N[2], 1, s);
    }
  }
};

}  // namespace
}  // namespace tdb
