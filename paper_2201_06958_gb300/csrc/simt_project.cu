// simt_project.cu - the projection of Eqs. 2.15/2.16 with the snapshot difference fused in,
// in float or double on the CUDA cores (the compute types without BF16 operands).
//
// One pass reads V_{k+1} and V_k once and leaves partial first contractions of
// dV = V_{k+1} - V_k over tiles of 128 points of mode 1 and `ti2` points of mode 2:
//   Z1 = dV x_1 A_1^T (summed over the tile's i1) and Z2 = dV x_2 A_2^T (over its i2),
// with ||dV||_W^2 and the finiteness check on the way; proj_finish.cuh contracts the rest.
//
// Bound: float by latency (12 warps an SM of one group after the other: loads, then products
// through shared memory), double by its arithmetic (two lanes per clock and SM).  256 x 128 x
// 512 float at ranks (11, 8, 16): 56 us, 53 with ||dV||^2 summed in single floats, which cost the
// norm its last bits (58 so with the sums of Z1 over the lanes formed by a butterfly of 31 shuffles
// and nothing fetched ahead), where difference, norm and the mode
// products that contract S points took 428 us; 126^3 double at (5, 5, 5): 87 us against 251
// us.  One CTA of eight warps per SM with the next rows prefetched into registers measured the
// same as three of four without.
#include <type_traits>

#include "proj_finish.cuh"
#include "simt_project.h"

namespace tdb {
namespace {

constexpr int SP_T1 = 128;            // i1 points of a tile: 32 lanes x 4
constexpr int SP_WARPS = 4;
constexpr int SP_THREADS = SP_WARPS * 32;
// Resident CTAs per SM: within 168 registers a thread in float; double needs 240.
template <typename T>
constexpr int kSpPerSm = sizeof(T) == 4 ? 3 : 2;
template <typename T>
constexpr int kSpCtas = kSpPerSm<T> * 152;

template <typename T>
struct SpParams {
  const T* Vn;
  const T* Vp;
  int N1, N2, nslice;
  int nq1, nq2, ti2;             // tile positions and the i2 points of a tile
  int cstep;                     // CTAs per tile position
  int r1, r2;
  const T* A1;                   // W_1 U_1 (N1 x r1), W_2 U_2 (N2 x r2)
  const T* A2;
  const double* w1;
  const double* w2;
  const double* wsl;
  T* Z1p;                        // [nq1][nslice][r1][N2]
  T* Z2p;                        // [nq2][nslice][r2][N1]
  double* npart;                 // per warp of the first rank block: [CTA][SP_WARPS]
  unsigned* flags;
  T dscale;
};

// Rows of a group (one butterfly of 32 sums is G rows x 32 / G ranks).
template <typename T>
struct SpCfg;
template <>
struct SpCfg<float> { static constexpr int G = 8; };
template <>
struct SpCfg<double> { static constexpr int G = 4; };

// Copies of an A_2 value in shared memory: float reads pairs (a, a) for its paired
// multiply-adds.  A warp's shared values: the differences of a group (float, rows SP_DLD
// apart), then its sums of Z2.
template <typename T>
constexpr int kSpDup = sizeof(T) == 4 ? 2 : 1;
constexpr int SP_DLD = SP_T1 + 4;
template <typename T>
constexpr int sp_warp_elems(int rb) {
  return sizeof(T) == 4 && rb * SP_T1 < SpCfg<float>::G * SP_DLD ? SpCfg<float>::G * SP_DLD : rb * SP_T1;
}

template <typename T, int RB>
constexpr size_t sp_smem(int ti2) {
  return sizeof(T) * ((size_t)RB * SP_T1 + (size_t)ti2 * RB * kSpDup<T> + (size_t)ti2 * kSpDup<T> + (size_t)RB * ti2 +
                      (size_t)SP_WARPS * sp_warp_elems<T>(RB));
}

__device__ __forceinline__ unsigned expo_bits(float v) { return __float_as_uint(v) & 0x7fffffffu; }
__device__ __forceinline__ unsigned expo_bits(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }
template <typename T>
constexpr unsigned kExpInf = sizeof(T) == 4 ? 0x7f800000u : 0x7ff00000u;

// A CTA keeps one tile position and walks the slices s0, s0 + cstep, ...; blockIdx.y takes
// RB ranks of each mode.  A warp owns ti2 / 8 rows (i2) of the tile, its lanes four i1 each,
// G rows at a time in registers:
//   Z2: four i1 x RB accumulators per lane, A_2's row read as a broadcast; the eight warps'
//       sums are added through shared memory at the end of the slice.
//   Z1: float: the group's differences are staged in shared memory and multiplied by A_1 as a
//       small matrix product, four rows x every fourth rank a lane.  Double: per group of
//       32 / G ranks the lane's sums over its four i1 of G rows are added over the 32 lanes by
//       a transposing butterfly (31 shuffles for 32 sums, lane l ends with row l % G, rank
//       l / G).  Either leaves through a shared tile.
// Every sum has a fixed order.  Several CTAs of four warps per SM cover the loads of one
// another (a warp's group is 8 KB).
template <typename T, int RB>
__global__ void __launch_bounds__(SP_THREADS, kSpPerSm<T>) k_sp_project(SpParams<T> P, int vec) {
  constexpr int G = SpCfg<T>::G, AG = 32 / G;
  extern __shared__ __align__(16) unsigned char sp_raw[];
  const int ti2 = P.ti2;
  T* A1s = (T*)sp_raw;                         // [RB][128]
  T* A2s = A1s + RB * SP_T1;                   // [ti2][RB], each value kSpDup times
  T* Z1s = A2s + ti2 * RB * kSpDup<T>;         // [RB][ti2]
  T* Z2s = Z1s + RB * ti2;                     // [4][RB][128]
  constexpr int ZW = sp_warp_elems<T>(RB);     // a warp's part of it
  T* w2s = Z2s + SP_WARPS * ZW;                // [ti2] (float: the weight in two floats)
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) fin_dep_launch();
  const int nq12 = P.nq1 * P.nq2;
  const int pos = blockIdx.x % nq12, q1 = pos % P.nq1, q2 = pos / P.nq1;
  const int s_first = blockIdx.x / nq12;
  const int r0 = blockIdx.y * RB;
  const int n1 = min(RB, P.r1 - r0), n2 = min(RB, P.r2 - r0);   // ranks of this block (may be <= 0)
  const int N1 = P.N1, N2 = P.N2, b1 = q1 * SP_T1, b2 = q2 * ti2;
  // i1 of slot j of this lane: four consecutive points, or every 32nd where the rows are not
  // 16-byte aligned (then each load is one value, consecutive over the lanes)
  auto i1_of = [&](int l, int j) { return b1 + (vec ? 4 * l + j : l + 32 * j); };
  for (int e = tid; e < RB * SP_T1; e += SP_THREADS) {
    const int a = e / SP_T1, x = e % SP_T1, i = i1_of(x >> 2, x & 3);
    A1s[e] = (a < n1 && i < N1) ? P.A1[i + (int64_t)N1 * (r0 + a)] : T(0);
  }
  for (int e = tid; e < RB * ti2; e += SP_THREADS) {
    const int b = e / ti2, x = e % ti2, i = b2 + x;
    const T a = (b < n2 && i < N2) ? P.A2[i + (int64_t)N2 * (r0 + b)] : T(0);
#pragma unroll
    for (int u = 0; u < kSpDup<T>; ++u) A2s[(x * RB + b) * kSpDup<T> + u] = a;
  }
  for (int x = tid; x < ti2; x += SP_THREADS) {
    const double w = b2 + x < N2 ? P.w2[b2 + x] : 0.0;
    if constexpr (sizeof(T) == 4) {
      w2s[2 * x] = (float)w;
      w2s[2 * x + 1] = (float)(w - (double)(float)w);
    } else {
      w2s[x] = w;
    }
  }
  T w1r[4];
  bool in1[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    in1[j] = i1_of(lane, j) < N1;
    w1r[j] = in1[j] ? (T)P.w1[i1_of(lane, j)] : T(0);
  }
  __syncthreads();
  const int wrows = ti2 / SP_WARPS, ngrp = (wrows + G - 1) / G;
  auto load = [&](int sl, int grp, T (&rn)[G][4], T (&rp)[G][4]) {
    const int64_t row0 = (int64_t)sl * N2 + b2 + warp * wrows + grp * G;
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const bool rin = grp * G + g < wrows && b2 + warp * wrows + grp * G + g < N2;
      const int64_t off = (row0 + g) * N1;
      if (vec) {
        Quad<T> x{T(0), T(0), T(0), T(0)}, y{T(0), T(0), T(0), T(0)};
        if (rin && in1[0]) {
          if constexpr (sizeof(T) == 4) {
            const float4 u = __ldcs((const float4*)(P.Vn + off + b1 + 4 * lane));
            const float4 v = __ldg((const float4*)(P.Vp + off + b1 + 4 * lane));
            x = Quad<T>{u.x, u.y, u.z, u.w};
            y = Quad<T>{v.x, v.y, v.z, v.w};
          } else {
            const double2 u0 = __ldcs((const double2*)(P.Vn + off + b1 + 4 * lane));
            const double2 v0 = __ldg((const double2*)(P.Vp + off + b1 + 4 * lane));
            x.x = u0.x; x.y = u0.y;
            y.x = v0.x; y.y = v0.y;
            if (in1[2]) {                  // (N1 even: a pair is in or out)
              const double2 u1 = __ldcs((const double2*)(P.Vn + off + b1 + 4 * lane + 2));
              const double2 v1 = __ldg((const double2*)(P.Vp + off + b1 + 4 * lane + 2));
              x.z = u1.x; x.w = u1.y;
              y.z = v1.x; y.w = v1.y;
            }
          }
        }
        rn[g][0] = x.x; rn[g][1] = x.y; rn[g][2] = x.z; rn[g][3] = x.w;
        rp[g][0] = y.x; rp[g][1] = y.y; rp[g][2] = y.z; rp[g][3] = y.w;
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const bool in = rin && in1[j];
          rn[g][j] = in ? __ldcs(P.Vn + off + i1_of(lane, j)) : T(0);
          rp[g][j] = in ? __ldg(P.Vp + off + i1_of(lane, j)) : T(0);
        }
      }
    }
  };
  // The next group's rows into L2 while this one is computed (a group is 12 000 cycles of its
  // warp): lane l takes 128 bytes of row l / 4 of both snapshots.
  auto fetch_l2 = [&](int sl, int grp) {
    constexpr int SEG = SP_T1 * (int)sizeof(T) / 128;        // 128-byte pieces of a row
#pragma unroll
    for (int u = lane; u < G * SEG; u += 32) {
      const int g = u / SEG, i = b1 + (u % SEG) * (128 / (int)sizeof(T)), x = warp * wrows + grp * G + g;
      if (grp * G + g < wrows && b2 + x < N2 && i < N1) {
        const int64_t off = ((int64_t)sl * N2 + b2 + x) * N1 + i;
        asm volatile("prefetch.global.L2 [%0];" ::"l"(P.Vn + off));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(P.Vp + off));
      }
    }
  };
  double acc_norm = 0.0;
  bool bad = false;
  for (int sl = s_first; sl < P.nslice; sl += P.cstep) {
    T acc2[RB][4];
#pragma unroll
    for (int b = 0; b < RB; ++b)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc2[b][j] = T(0);
    // ||dV||_W^2 of this lane's points of the slice: the four points of a row in T, everything
    // after that in double (float: in a pair of floats)
    typename std::conditional<sizeof(T) == 4, FloatPair, double>::type nrm{};
    for (int grp = 0; grp < ngrp; ++grp) {
      const int x0 = warp * wrows + grp * G;               // first row of the group within the tile
      T d[G][4];
      {
        T rn[G][4], rp[G][4];
        load(sl, grp, rn, rp);
        if (grp + 1 < ngrp) fetch_l2(sl, grp + 1);
        else if (sl + P.cstep < P.nslice) fetch_l2(sl + P.cstep, 0);
        bool odd = false;                                  // a row sum that is not finite
#pragma unroll
        for (int g = 0; g < G; ++g) {
          T q = T(0);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            d[g][j] = rn[g][j] - rp[g][j];
            q = fma(w1r[j] * d[g][j], d[g][j], q);
          }
          odd |= expo_bits(q) >= kExpInf<T>;
          if (grp * G + g < wrows) {
            if constexpr (sizeof(T) == 4) nrm.add_product(w2s[2 * (x0 + g)], w2s[2 * (x0 + g) + 1], q);
            else nrm = fma(w2s[x0 + g], q, nrm);
          }
        }
        if (odd) {                                         // ... by a difference, or only by its square
#pragma unroll
          for (int g = 0; g < G; ++g)
#pragma unroll
            for (int j = 0; j < 4; ++j) bad |= expo_bits(d[g][j]) >= kExpInf<T>;
        }
      }
      // Z2: this lane's four i1, RB ranks of mode 2
#pragma unroll
      for (int g = 0; g < G; ++g) {
        if (grp * G + g >= wrows) break;
        const Quad<T>* a2 = reinterpret_cast<const Quad<T>*>(A2s + (x0 + g) * RB * kSpDup<T>);
        if constexpr (sizeof(T) == 4) {
          const float2 d0 = make_float2(d[g][0], d[g][1]), d1 = make_float2(d[g][2], d[g][3]);
#pragma unroll
          for (int b2x = 0; b2x < RB / 2; ++b2x) {
            if (b2x % 2 == 0 && 2 * b2x >= n2) break;
            const Quad<T> a = a2[b2x];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              T (&c)[4] = acc2[2 * b2x + u];
              const float2 aa = u ? make_float2(a.z, a.w) : make_float2(a.x, a.y);
              const float2 lo = __ffma2_rn(d0, aa, make_float2(c[0], c[1]));
              const float2 hi = __ffma2_rn(d1, aa, make_float2(c[2], c[3]));
              c[0] = lo.x; c[1] = lo.y; c[2] = hi.x; c[3] = hi.y;
            }
          }
        } else {
#pragma unroll
          for (int b4 = 0; b4 < RB / 4; ++b4) {
            if (4 * b4 >= n2) break;
            const Quad<T> a = a2[b4];
            const T av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
            for (int u = 0; u < 4; ++u)
              if (4 * b4 + u < n2)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc2[4 * b4 + u][j] = fma(d[g][j], av[u], acc2[4 * b4 + u][j]);
          }
        }
      }
      if constexpr (sizeof(T) == 4) {
        // Z1: a small matrix product.  The group's G x 128 differences are staged for the warp;
        // lane (kq, rg, ag) sums every fourth run of four i1 for four rows and the ranks ag,
        // ag + 4, ..., and the four kq lanes' sums are added by a transposing exchange.
        T* ds = Z2s + warp * ZW;
        __syncwarp();
#pragma unroll
        for (int g = 0; g < G; ++g)
          *reinterpret_cast<float4*>(ds + g * SP_DLD + 4 * lane) = make_float4(d[g][0], d[g][1], d[g][2], d[g][3]);
        __syncwarp();
        const int kq = lane & 3, rg = (lane >> 2) & 1, ag = lane >> 3;
        float2 z[RB / 4][4];
#pragma unroll
        for (int t = 0; t < RB / 4; ++t)
#pragma unroll
          for (int r = 0; r < 4; ++r) z[t][r] = make_float2(0.f, 0.f);
#pragma unroll 2
        for (int q = kq; q < SP_T1 / 4; q += 4) {
          float4 x[4];
#pragma unroll
          for (int r = 0; r < 4; ++r) x[r] = *reinterpret_cast<const float4*>(ds + (4 * rg + r) * SP_DLD + 4 * q);
#pragma unroll
          for (int t = 0; t < RB / 4; ++t) {
            if (4 * t >= n1) break;
            const float4 a = *reinterpret_cast<const float4*>(A1s + (ag + 4 * t) * SP_T1 + 4 * q);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              z[t][r] = __ffma2_rn(make_float2(x[r].x, x[r].y), make_float2(a.x, a.y), z[t][r]);
              z[t][r] = __ffma2_rn(make_float2(x[r].z, x[r].w), make_float2(a.z, a.w), z[t][r]);
            }
          }
        }
#pragma unroll
        for (int t = 0; t < RB / 4; ++t) {
          if (4 * t >= n1) break;
          T v[4];
#pragma unroll
          for (int r = 0; r < 4; ++r) v[r] = z[t][r].x + z[t][r].y;
#pragma unroll
          for (int o = 2; o > 0; o >>= 1) {
            const bool up = kq & o;
#pragma unroll
            for (int i = 0; i < o; ++i) {
              const T keep = up ? v[i + o] : v[i], send = up ? v[i] : v[i + o];
              v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
          }
          const int g = 4 * rg + kq;
          if (grp * G + g < wrows) Z1s[(ag + 4 * t) * ti2 + x0 + g] = v[0];
        }
      } else {
        // Z1: AG ranks of mode 1 at a time over the G rows
#pragma unroll
        for (int ag = 0; ag < RB / AG; ++ag) {
          if (AG * ag >= n1) break;
          T v[32];
#pragma unroll
          for (int aa = 0; aa < AG; ++aa) {
            if (AG * ag + aa >= n1) {
#pragma unroll
              for (int g = 0; g < G; ++g) v[g + G * aa] = T(0);
              continue;
            }
            const Quad<T> a = *reinterpret_cast<const Quad<T>*>(A1s + (AG * ag + aa) * SP_T1 + 4 * lane);
#pragma unroll
            for (int g = 0; g < G; ++g)
              v[g + G * aa] = fma(d[g][3], a.w, fma(d[g][2], a.z, fma(d[g][1], a.y, d[g][0] * a.x)));
          }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            const bool up = lane & o;
#pragma unroll
            for (int i = 0; i < o; ++i) {
              const T keep = up ? v[i + o] : v[i], send = up ? v[i] : v[i + o];
              v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
          }
          const int g = lane % G, a = AG * ag + lane / G;
          if (grp * G + g < wrows) Z1s[a * ti2 + x0 + g] = v[0];
        }
      }
    }
    if (r0 == 0) {
      if constexpr (sizeof(T) == 4) acc_norm += P.wsl[sl] * nrm.value();
      else acc_norm += P.wsl[sl] * nrm;
    }
    // the slice's partials leave: Z1 as it is, Z2 summed over the warps in order
    __syncwarp();
#pragma unroll
    for (int b = 0; b < RB; ++b)
      *reinterpret_cast<Quad<T>*>(Z2s + warp * ZW + b * SP_T1 + 4 * lane) =
          Quad<T>{acc2[b][0], acc2[b][1], acc2[b][2], acc2[b][3]};
    __syncthreads();
    for (int e = tid; e < n1 * ti2; e += SP_THREADS) {
      const int a = e / ti2, x = e % ti2;
      if (b2 + x < N2) P.Z1p[(((int64_t)q1 * P.nslice + sl) * P.r1 + r0 + a) * N2 + b2 + x] = Z1s[e] * P.dscale;
    }
    for (int e = tid; e < n2 * SP_T1; e += SP_THREADS) {
      const int b = e / SP_T1, x = e % SP_T1;
      const int at = vec ? x : 4 * (x & 31) + (x >> 5);
      T s = Z2s[b * SP_T1 + at];
#pragma unroll
      for (int w = 1; w < SP_WARPS; ++w) s += Z2s[w * ZW + b * SP_T1 + at];
      if (b1 + x < N1) P.Z2p[(((int64_t)q2 * P.nslice + sl) * P.r2 + r0 + b) * N1 + b1 + x] = s * P.dscale;
    }
    __syncthreads();
  }
  if (r0 == 0) {
    if (bad) atomicOr(P.flags, kFlagNonFinite);
    const double t = warp_sum(acc_norm);
    if (lane == 0) P.npart[(int64_t)blockIdx.x * SP_WARPS + warp] = t * (double)P.dscale * (double)P.dscale;
  }
}

// The split of a projection: the tallest tile (i2 points, at most 128) that still gives four
// tiles to every resident CTA, so that the last wave costs little; not below the rows one
// pass of a CTA takes, nor so low that mode 2 has more tiles than the finish loads at once.
// Every tile position is walked by the same number of CTAs.
struct SpShape {
  int nq1, nq2, ti2, cstep, nblk, rb;
};
template <typename T>
SpShape sp_shape(const int64_t* N, const int* r, int64_t nslice) {
  SpShape h;
  const int rmax = std::max(r[0], r[1]);
  if (sizeof(T) == 8) {
    h.rb = 8;
    h.nblk = (rmax + 7) / 8;
  } else {
    h.nblk = (rmax + 15) / 16;
    h.rb = (((rmax + h.nblk - 1) / h.nblk) + 3) & ~3;
  }
  h.nq1 = (int)((N[0] + SP_T1 - 1) / SP_T1);
  const int low = SP_WARPS * SpCfg<T>::G;
  h.ti2 = 128;
  while (h.ti2 > low && (h.ti2 / 2) * FS_NQ_MAX >= N[1] &&
         (N[1] <= h.ti2 / 2 || h.nq1 * ((N[1] + h.ti2 - 1) / h.ti2) * nslice * h.nblk < 4 * kSpCtas<T>))
    h.ti2 /= 2;
  h.nq2 = (int)((N[1] + h.ti2 - 1) / h.ti2);
  const int64_t per = (int64_t)h.nq1 * h.nq2 * h.nblk;
  h.cstep = (int)std::max<int64_t>(1, std::min<int64_t>(nslice, kSpCtas<T> / per));
  return h;
}

int64_t slices(int p, const int64_t* N) {
  int64_t v = 1;
  for (int n = 2; n < p; ++n) v *= N[n];
  return v;
}

// Most tiles along mode 2 that sp_shape makes: with one rank block (more blocks fill the SMs with
// taller tiles).
template <typename T>
int64_t sp_tiles2_max(const int64_t* N, int64_t nslice) {
  const int r[2] = {1, 1};
  return sp_shape<T>(N, r, nslice).nq2;
}

// Points that the tiles of a pass cover, over the tensor's (with one rank block).
template <typename T>
double sp_padding(int p, const int64_t* N) {
  const int r[2] = {1, 1};
  const SpShape h = sp_shape<T>(N, r, slices(p, N));
  return (double)h.nq1 * SP_T1 / N[0] * ((double)h.nq2 * h.ti2 / N[1]);
}

template <typename T, int RB>
void sp_launch(const SpParams<T>& P, const SpShape& h, int vec, cudaStream_t s) {
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_sp_project<T, RB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sp_smem<T, RB>(128));
    attr = true;
  }
  k_sp_project<T, RB><<<dim3(h.nq1 * h.nq2 * h.cstep, h.nblk), SP_THREADS, sp_smem<T, RB>(h.ti2), s>>>(P, vec);
  count_launch();
}

}  // namespace

// The pass against the mode products, a step of 800 sizes each way (us, pass to products):
// Float: faster nearly everywhere (256 x 128 x 512 at ranks (11, 8, 16) 60 to 430, 32^3 (3) 65 to 69);
//   a short mode 2 of four wastes its tiles (64 x 3 x 64 x 64 (3) 193 to 114, 3 x 3 x 3 x 20 000 (8)
//   2263 to 652; 64 x 64 x 3 x 64 (3) 77 to 110), and so does one of three with many slices (5 x 5 x
//   42 223 (5) 1004 to 726, 35 x 4 x 7332 (27) 459 to 294; 31 x 9 x 738 (9) 108 to 125): the line at
//   20 points, and 4096 slices with three modes.
// Double, two modes: a warp's lanes lie along mode 1 (20 x 50 000 872 to 446, 7 x 100 000 1676 to 810;
//   200 x 200 80 to 195, 50 000 x 20 233 to 1769): the line lay between 48 and 55 points.
// Double, three modes: a last mode of up to 64 points has a cheaper product (64^3 at ranks 3 and 16 86
//   to 89 and 220 to 182, 400 x 400 x 8 (8) 231 to 157; 96^3 (3, 16) 114 to 269 and 297 to 459, 126^3 (5)
//   100 to 410).  Above that, tiles that are mostly padding cost their arithmetic (13 x 4 x 1928 (10)
//   634 to 156 at 39 times the points, 19 x 9 x 10 281 (6) 1557 to 5554 at twelve); beside a mode 2 that
//   fills its tiles a short mode 1 does already (41 x 582 x 116 (16) 1645 to 1063, 224 x 332 x 97 (4) 412
//   to 660); and a mode 1 of seven tiles and more is cheap for the products (9633 x 4 x 85 (6) 987
//   to 834).
// Double, four modes: the finish forms r_3 r_4 outputs a slice with double's arithmetic (40 x 40 x 40 x 8
//   (8) 375 to 185); even at 1.5 times the points.
template <typename T>
bool sp_worth(int p, const int64_t* N) {
  if (sizeof(T) == 4) return p == 2 || N[1] > 20 || (p == 3 && N[2] <= 4096);
  if (p == 2) return N[0] >= 52;
  if (p == 3) return N[2] > 64 && (N[1] <= 256 ? N[0] <= 7 * SP_T1 && sp_padding<T>(p, N) <= 30 : N[0] >= 48);
  return sp_padding<T>(p, N) <= 1.5;
}
template bool sp_worth<float>(int, const int64_t*);
template bool sp_worth<double>(int, const int64_t*);

bool sp_supported(int p, const int* r) { return finish_outputs(p, r) <= FS_JMAX; }

void sp_carve_weights(SpPlan& plan, Carver& cv, int p, const int64_t* N) {
  plan.wsl = cv.take<double>((size_t)slices(p, N));
}

template <typename T>
void sp_carve_pass(SpPlan& plan, Carver& cv, int p, const int64_t* N, const int* cap) {
  const int64_t ns = slices(p, N);
  const int64_t nq1 = (N[0] + SP_T1 - 1) / SP_T1, nq2 = sp_tiles2_max<T>(N, ns);
  plan.z1p = cv.take<T>((size_t)(nq1 * ns * N[1] * cap[0]));
  plan.z2p = cv.take<T>((size_t)(nq2 * ns * N[0] * cap[1]));
  plan.npart = cv.take<double>((size_t)std::max<int64_t>(kSpCtas<T>, nq1 * nq2) * SP_WARPS);
  plan.fpart_cap = finish_split_elems<T>(p, N, cap);
  plan.fpart = cv.take<T>(plan.fpart_cap);
  plan.wrest = p == 4 ? cv.take<T>((size_t)cap[0] * cap[1] * ns) : nullptr;
}
template void sp_carve_pass<float>(SpPlan&, Carver&, int, const int64_t*, const int*);
template void sp_carve_pass<double>(SpPlan&, Carver&, int, const int64_t*, const int*);

void sp_prepare(SpPlan& plan, int p, const int64_t* N, const double* const* w, cudaStream_t s) {
  const int64_t ns = slices(p, N);
  k_slice_weights<<<(unsigned)((ns + 255) / 256), 256, 0, s>>>(p, p >= 3 ? w[2] : nullptr, p >= 3 ? (int)N[2] : 1,
                                                              p >= 4 ? w[3] : nullptr, p >= 4 ? (int)N[3] : 1,
                                                              plan.wsl);
  count_launch();
}

template <typename T>
tdb_status sp_project(SpPlan& plan, const T* Vn, const T* Vp, int p, const int64_t* N, const int* r,
                      const void* const* A, const double* const* w, T* Z1, T* const* Y, double* dv2, unsigned* flags,
                      cudaStream_t s, cudaEvent_t* evm, std::string& err, T dscale) {
  const int64_t ns = slices(p, N);
  const SpShape h = sp_shape<T>(N, r, ns);
  SpParams<T> P;
  P.Vn = Vn;
  P.Vp = Vp;
  P.N1 = (int)N[0];
  P.N2 = (int)N[1];
  P.nslice = (int)ns;
  P.nq1 = h.nq1;
  P.nq2 = h.nq2;
  P.ti2 = h.ti2;
  P.cstep = h.cstep;
  P.r1 = r[0];
  P.r2 = r[1];
  P.A1 = (const T*)A[0];
  P.A2 = (const T*)A[1];
  P.w1 = w[0];
  P.w2 = w[1];
  P.wsl = plan.wsl;
  P.Z1p = (T*)plan.z1p;
  P.Z2p = (T*)plan.z2p;
  P.npart = plan.npart;
  P.flags = flags;
  P.dscale = dscale;
  // 16-byte loads where every row of both snapshots starts on a 16-byte boundary
  const int vec = (N[0] * sizeof(T)) % 16 == 0 && (((uintptr_t)Vn | (uintptr_t)Vp) & 15) == 0;
  if (evm) record_timing_event(evm[0], s);
  if constexpr (sizeof(T) == 8) {
    sp_launch<T, 8>(P, h, vec, s);
  } else {
    if (h.rb <= 4) sp_launch<T, 4>(P, h, vec, s);
    else if (h.rb <= 8) sp_launch<T, 8>(P, h, vec, s);
    else if (h.rb <= 12) sp_launch<T, 12>(P, h, vec, s);
    else sp_launch<T, 16>(P, h, vec, s);
  }
  if (evm) record_timing_event(evm[1], s);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    err = std::string("projection launch: ") + cudaGetErrorString(e);
    return TDB_ERR_CUDA;
  }
  Finish<T> fin;
  fin.setup(p, N, r, A, Z1, (T*)plan.z1p, (T*)plan.z2p, h.nq1, h.nq2, (T*)plan.wrest, Y, (T*)plan.fpart,
            plan.fpart_cap, plan.npart, dv2, s);
  fin.f.nnp = h.nq1 * h.nq2 * h.cstep * SP_WARPS;
  fin.launch(fin.nsplit_for(FS_CTAS));
  fin.launch_rest(N, r, A, Y);
  e = cudaGetLastError();
  if (e != cudaSuccess) {
    err = std::string("projection finish: ") + cudaGetErrorString(e);
    return TDB_ERR_CUDA;
  }
  return TDB_OK;
}
template tdb_status sp_project<float>(SpPlan&, const float*, const float*, int, const int64_t*, const int*,
                                      const void* const*, const double* const*, float*, float* const*, double*,
                                      unsigned*, cudaStream_t, cudaEvent_t*, std::string&, float);
template tdb_status sp_project<double>(SpPlan&, const double*, const double*, int, const int64_t*, const int*,
                                       const void* const*, const double* const*, double*, double* const*, double*,
                                       unsigned*, cudaStream_t, cudaEvent_t*, std::string&, double);

}  // namespace tdb
