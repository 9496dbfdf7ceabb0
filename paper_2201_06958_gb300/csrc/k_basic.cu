// k_basic.cu - elementwise kernels, weighted norms and the generic n-mode product.
//
// The n-mode product (Sec. 2.1) out = in x_n M, with M of shape J x K, is taken on
// the view in = (L, K, Q), out = (L, J, Q) (column-major, l fastest), where
// L = prod of the sizes before mode n and Q = prod of the sizes after it:
//     out[l + L (j + J q)] = sum_k M[j sMj + k sMk] in[l + L (k + K q)].
// It serves the unfused projection (M = A_n^T = (W_n U_n)^T, Eqs. 2.15/2.16),
// the reconstruction (M = U_n, Eq. 2.5) and the core compensation (M = R_n).
#include "common.cuh"
#include "kernels.h"

#include <atomic>
#include <type_traits>

namespace tdb {

static std::atomic<long long> g_launches{0};
void count_launch(int n) { g_launches.fetch_add(n, std::memory_order_relaxed); }
long long launches_so_far() { return g_launches.load(std::memory_order_relaxed); }

// ---------------------------------------------------------------------------
// Elementwise
// ---------------------------------------------------------------------------

// Everything of a state (T, U_n) that other kernels read beside it, in one launch: the core and
// the bases in the compute type (float types) and, if asked for, A_n = W_n U_n (Eq. 2.17); with
// `src` the state is first taken from there (T, then U_1 .. U_p, as a saved state holds it).
// One launch instead of two or three per mode: a state load is launches and copies.
template <typename T>
__global__ void __launch_bounds__(256) k_state_views(StateViews v) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < v.total; e += (int64_t)gridDim.x * blockDim.x) {
    if (e < v.nT) {
      const double x = v.src ? v.src[e] : v.T[e];
      if (v.src) v.T[e] = x;
      if (v.Tcore != v.T) ((T*)v.Tcore)[e] = (T)x;
      continue;
    }
    int64_t k = e - v.nT;
    int n = 0;
    while (k >= v.N[n] * v.r[n]) { k -= v.N[n] * v.r[n]; ++n; }
    const double x = v.src ? v.src[e] : v.U[n][k];
    if (v.src) v.U[n][k] = x;
    ((T*)v.Uc[n])[k] = (T)x;
    if (v.bases) ((T*)v.A[n])[k] = (T)(v.w[n][k % v.N[n]] * x);
  }
}
// The reverse: T, U_1 .. U_p one after another, for one copy to the host.
__global__ void __launch_bounds__(256) k_state_pack(StateViews v, double* __restrict__ out) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < v.total; e += (int64_t)gridDim.x * blockDim.x) {
    int64_t k = e - v.nT;
    int n = 0;
    if (k >= 0)
      while (k >= v.N[n] * v.r[n]) { k -= v.N[n] * v.r[n]; ++n; }
    out[e] = k < 0 ? v.T[e] : v.U[n][k];
  }
}
template <typename T>
void launch_state_views(const StateViews& v, cudaStream_t s) {
  const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((v.total + 255) / 256, 152 * 8));
  k_state_views<T><<<blocks, 256, 0, s>>>(v); count_launch();
}
template void launch_state_views<float>(const StateViews&, cudaStream_t);
template void launch_state_views<double>(const StateViews&, cudaStream_t);
void launch_state_pack(const StateViews& v, double* out, cudaStream_t s) {
  const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((v.total + 255) / 256, 152 * 8));
  k_state_pack<<<blocks, 256, 0, s>>>(v, out); count_launch();
}

template <typename Ts, typename Td>
__global__ void k_cast(const Ts* __restrict__ a, Td* __restrict__ b, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    b[i] = (Td)a[i];
}
template <typename Ts, typename Td>
void launch_cast(const Ts* a, Td* b, int64_t n, cudaStream_t s) {
  int blocks = (int)std::min<int64_t>((n + 255) / 256, 1024);
  if (blocks < 1) blocks = 1;
  k_cast<Ts, Td><<<blocks, 256, 0, s>>>(a, b, n); count_launch();
}
template void launch_cast<float, double>(const float*, double*, int64_t, cudaStream_t);

// ---------------------------------------------------------------------------
// The snapshot difference out = scale (a - b) (scale 1, or a central difference's) and its
// weighted squared norm (Eq. 2.2 with the quadrature of Eq. 2.17) in one pass, for the mode
// products' route of the projection:
//   sum_i w_1(i_1) ... w_p(i_p) out[i]^2
// A warp per mode-1 column; a lane's products of a column are added in double (float: in a pair of
// floats) and weighted by the column's prod_{m>1} w_m in double (double: from `wcol`).  Deterministic:
// warp and CTA partials in a fixed order, added by the last CTA to finish (`counter` is zero
// before and after).  64^3 double from a cold cache: 12.7 us, as difference, norm and
// sum apart 23.7 us.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) k_diff_norm(const T* __restrict__ a, const T* __restrict__ b, T* __restrict__ out,
                                                   int N1, unsigned ncol, T scale, const T* __restrict__ w1,
                                                   const T* __restrict__ wcol, WeightView wv,
                                                   double* __restrict__ partial,
                                                   unsigned* __restrict__ counter, double* __restrict__ norm2,
                                                   unsigned* flags) {
  __shared__ double sh[32];
  __shared__ bool last;
  const int lane = threadIdx.x & 31;
  const unsigned nw = gridDim.x * (blockDim.x >> 5);
  double acc = 0.0;
  bool bad = false;
  for (unsigned c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); c < ncol; c += nw) {
    const size_t o = (size_t)N1 * c;
    typename std::conditional<sizeof(T) == 4, FloatPair, double>::type s{};
    for (int i = lane; i < N1; i += 32) {
      const T d = (a[o + i] - b[o + i]) * scale;
      out[o + i] = d;
      bad |= !isfinite(d);
      if constexpr (sizeof(T) == 4) s.add((w1[i] * d) * d);
      else s = fma(w1[i] * d, d, s);
    }
    if constexpr (sizeof(T) == 4) {
      double wc = 1.0;
      unsigned rem = c;
      for (int m = 1; m < wv.p; ++m) {
        const unsigned nm = (unsigned)wv.N[m];
        wc *= wv.w[m][rem % nm];
        rem /= nm;
      }
      acc = fma(wc, s.value(), acc);
    } else {
      acc = fma(wcol[c], s, acc);
    }
  }
  acc = block_sum(acc, sh);
  if (bad && flags) atomicOr(flags, kFlagNonFinite);
  if (threadIdx.x == 0) {
    partial[blockIdx.x] = acc;
    __threadfence();
    last = (atomicAdd(counter, 1u) == gridDim.x - 1);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double t = 0.0;
  for (int k = threadIdx.x; k < (int)gridDim.x; k += blockDim.x) t += __ldcg(&partial[k]);
  t = block_sum(t, sh);
  if (threadIdx.x == 0) {
    *norm2 = t;
    atomicExch(counter, 0u);
  }
}

template <typename T>
void launch_diff_norm(const T* a, const T* b, T* out, int N1, int64_t ncol, T scale, const T* w1, const T* wcol,
                      const WeightView& wv,
                      double* partial, unsigned* counter, int nblocks, double* norm2, unsigned* flags, cudaStream_t s) {
  const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(nblocks, (ncol + 7) / 8));
  k_diff_norm<T><<<blocks, 256, 0, s>>>(a, b, out, N1, (unsigned)ncol, scale, w1, wcol, wv, partial, counter, norm2,
                                     flags);
  count_launch();
}
template void launch_diff_norm<float>(const float*, const float*, float*, int, int64_t, float, const float*,
                                      const float*, const WeightView&, double*, unsigned*, int, double*, unsigned*, cudaStream_t);
template void launch_diff_norm<double>(const double*, const double*, double*, int, int64_t, double, const double*,
                                       const double*, const WeightView&, double*, unsigned*, int, double*, unsigned*, cudaStream_t);

// Exact error of Eq. 2.20 without materialising V^TDB: with H = T x_2 U_2 ... x_p U_p
// (r_1 x N_2 x ... x N_p), every mode-1 column of the reconstruction is U_1 H[:, c].
// Lane l of a warp owns rows i0 + R l .. i0 + R l + R - 1 of a block of 32 R rows, with U_1 of
// those rows (R x r_1) and w_1 in registers, and walks a contiguous range of columns c.  Its R
// rows of each column arrive by cp.async in a ring of D slots (D columns in flight per warp,
// read back by the lane that copied them: no barrier); H and w_c come 32 columns at a time, H by
// cp.async into one of two halves of shared rows padded to RM (zeros past r_1), w_c a column per
// lane.  Per column
// the lane forms U_1 H[:, c] for its rows and the weighted squared difference; w_c times it
// goes into a sum of the compute type that is added to the double accumulator every D columns.
// The last CTA to finish adds the per-CTA partials in a fixed order and writes *out (no second
// launch); `counter` is zero before and after.  Double runs at 64 cycles per instruction and
// sub-partition, so there only the r_1 products that exist are formed (float takes all RM, in
// pairs).  Measured from a cold cache: 256 x 128 x 512 float at r_1 = 11, 25.4 us (26.7 with H
// through registers, which spilled above rank 12, and single products; 32 with a column's H
// and w_c copied beside its rows and two warp barriers a column); 126^3 double at
// r_1 = 5, 54 us (8 double operations a point: 30 us at the issue rate), where a warp per column
// with U_1 in shared memory and H[:, c] by shuffles took 156 us.
constexpr int RE_D = 8;           // columns in flight per warp
template <int N>
using IntC = std::integral_constant<int, N>;
template <int BYTES>
__device__ __forceinline__ void cp_async_n(void* dst, const void* src, bool valid) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(valid ? 16 : 0) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %3, %2;" ::"r"(d), "l"(src), "r"(valid ? BYTES : 0), "n"(BYTES)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// N consecutive values from 16-byte aligned (N sizeof(T) >= 16) shared memory
template <typename T, int N>
__device__ __forceinline__ void lds_run(const T* p, T* v) {
  if constexpr (N * sizeof(T) % 16 == 0) {
    constexpr int per = 16 / sizeof(T);
#pragma unroll
    for (int i = 0; i < N / per; ++i) {
      if constexpr (sizeof(T) == 4) {
        const float4 t = reinterpret_cast<const float4*>(p)[i];
        v[4 * i] = t.x; v[4 * i + 1] = t.y; v[4 * i + 2] = t.z; v[4 * i + 3] = t.w;
      } else {
        const double2 t = reinterpret_cast<const double2*>(p)[i];
        v[2 * i] = t.x; v[2 * i + 1] = t.y;
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = p[i];
  }
}

// Columns of a chunk: 32, or 16 where two chunks of 32 would leave one CTA per SM.
template <typename T, int RM>
constexpr int kChunk = sizeof(T) * RM <= 128 ? 32 : 16;

// A chunk of columns of an r1 x ncol matrix (contiguous) on their way by cp.async into a warp's
// shared rows of RM.  Value e goes to row e / r1, entry e % r1 (stepped, not divided).
template <typename T, int RM>
__device__ __forceinline__ void fetch_columns(T* dst, const T* __restrict__ H, int r1, unsigned c, unsigned c_hi,
                                              int lane) {
  const int nv = c < c_hi ? r1 * (int)min((unsigned)kChunk<T, RM>, c_hi - c) : 0;
  const T* src = H + (size_t)r1 * (nv ? c : 0);
  const int dq = 32 / r1, dr = 32 - dq * r1, q = lane / r1;
  int rem = lane - q * r1, off = q * RM + rem;
#pragma unroll 1
  for (int e = lane; e < kChunk<T, RM> * r1; e += 32) {       // (unrolled, its offsets would stay in registers)
    cp_async_n<sizeof(T)>(dst + off, e < nv ? src + e : src, e < nv);
    off += dq * RM + dr;
    rem += dr;
    if (rem >= r1) { rem -= r1; off += RM - r1; }
  }
}

// U_1 of a lane's R rows in registers, and its product with one column of H.  Float: paired
// multiply-adds over (a, a + 1), the even and the odd terms' sums added last; double: only the
// r_1 products that exist.
template <typename T, int R, int RM>
struct RowBlock {
  T u[R][RM];
  __device__ __forceinline__ void load(const T* __restrict__ U1, int i0, int N1, int r1) {
#pragma unroll
    for (int q = 0; q < R; ++q)
#pragma unroll
      for (int a = 0; a < RM; ++a) u[q][a] = (i0 + q < N1 && a < r1) ? U1[i0 + q + (size_t)N1 * a] : T(0);
  }
  __device__ __forceinline__ void times(const T* h, int r1, T* rec) const {
    if constexpr (sizeof(T) == 4) {
      float2 acc[R];
#pragma unroll
      for (int q = 0; q < R; ++q) acc[q] = make_float2(0.f, 0.f);
#pragma unroll
      for (int a4 = 0; a4 < RM / 4; ++a4) {
        const float4 x = reinterpret_cast<const float4*>(h)[a4];
#pragma unroll
        for (int q = 0; q < R; ++q)
          acc[q] = __ffma2_rn(make_float2(u[q][4 * a4], u[q][4 * a4 + 1]), make_float2(x.x, x.y), acc[q]);
#pragma unroll
        for (int q = 0; q < R; ++q)
          acc[q] = __ffma2_rn(make_float2(u[q][4 * a4 + 2], u[q][4 * a4 + 3]), make_float2(x.z, x.w), acc[q]);
      }
#pragma unroll
      for (int q = 0; q < R; ++q) rec[q] = acc[q].x + acc[q].y;
    } else {
      T x[RM];
      lds_run<T, RM>(h, x);
#pragma unroll
      for (int q = 0; q < R; ++q) rec[q] = T(0);
#pragma unroll
      for (int a = 0; a < RM; ++a)
        if (a < r1)
#pragma unroll
          for (int q = 0; q < R; ++q) rec[q] = fma(u[q][a], x[a], rec[q]);
    }
  }
};

template <typename T, int R, int RM>
__global__ void __launch_bounds__(256, 2) k_recon_err_rows(const T* __restrict__ V, const T* __restrict__ U1,
                                                         const T* __restrict__ H, int r1, int N1, unsigned ncol,
                                                         const T* __restrict__ w1, const T* __restrict__ wcol,
                                                         int vec, double* __restrict__ partial,
                                                         unsigned* __restrict__ counter, double* __restrict__ out,
                                                         unsigned* flags, const int* __restrict__ gate) {
  if (gate && *gate == 0) return;          // the estimator ruled this evaluation out
  constexpr int CC = kChunk<T, RM>;
  extern __shared__ __align__(16) unsigned char ring_raw[];
  __shared__ double sh[32];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  T* ring = (T*)ring_raw + (size_t)wib * (RE_D * 32 * R + 2 * CC * RM) + R * lane;     // this lane's rows of slot 0
  T* hs = (T*)ring_raw + (size_t)wib * (RE_D * 32 * R + 2 * CC * RM) + RE_D * 32 * R;  // two chunks of H
  for (int e = lane; e < 2 * CC * RM; e += 32) hs[e] = T(0);
  const int nrb = (N1 + 32 * R - 1) / (32 * R);
  const unsigned gw = blockIdx.x * (blockDim.x >> 5) + wib, tw = gridDim.x * (blockDim.x >> 5);
  const unsigned wpr = tw >= (unsigned)nrb ? tw / nrb : 1u;   // warps per row block
  double acc = 0.0;
  bool bad = false;
  const unsigned kk = gw % wpr;
  const unsigned c_lo = (unsigned)((uint64_t)ncol * kk / wpr), c_hi = (unsigned)((uint64_t)ncol * (kk + 1) / wpr);
  // (a row block per group of wpr warps; the outer loop only where there are fewer warps than blocks)
  for (unsigned rb = gw / wpr; rb < (unsigned)nrb && c_lo < c_hi; rb += (tw >= (unsigned)nrb ? (unsigned)nrb : tw)) {
    const int i0 = (int)rb * 32 * R + R * lane;
    const bool rows_in = i0 < N1;
    const T* vsrc = V + (size_t)N1 * c_lo + (rows_in ? i0 : 0);   // the next column to issue
    unsigned cnext = c_lo;
    auto issue = [&](int sl) {
      const bool in = cnext < c_hi;
      T* dst = ring + sl * 32 * R;
      if (vec) {
        cp_async_n<R * sizeof(T)>(dst, vsrc, in && rows_in);
      } else {
#pragma unroll
        for (int q = 0; q < R; ++q)
          cp_async_n<sizeof(T)>(dst + q, vsrc + (i0 + q < N1 ? q : 0), in && i0 + q < N1);
      }
      cp_async_commit();
      ++cnext;
      if (cnext < c_hi) vsrc += N1;          // (past the end: zero bytes from the last column)
    };
    __syncwarp();                            // hs cleared, and the row block before is done with it
    fetch_columns<T, RM>(hs, H, r1, c_lo, c_hi, lane);
#pragma unroll
    for (int t = 0; t < RE_D; ++t) issue(t);
    T wn = lane < CC && c_lo + lane < c_hi ? __ldg(&wcol[c_lo + lane]) : T(0);
    RowBlock<T, R, RM> ub;
    ub.load(U1, i0, N1, r1);
    T wr[R];
#pragma unroll
    for (int q = 0; q < R; ++q) wr[q] = i0 + q < N1 ? w1[i0 + q] : T(0);
    T csum = T(0);
    int par = 0;                             // the half of hs that holds this chunk
    for (unsigned c0 = c_lo; c0 < c_hi; c0 += CC, par ^= 1) {
      // this chunk's H is in the group of the first column issued after it: older than the
      // RE_D - 1 that may be open
      cp_async_wait<RE_D - 1>();
      const T wl = wn;
      __syncwarp();
      fetch_columns<T, RM>(hs + CC * RM * (par ^ 1), H, r1, c0 + CC, c_hi, lane);
      const T* hc = hs + CC * RM * par;
      wn = lane < CC && c0 + CC + lane < c_hi ? __ldg(&wcol[c0 + CC + lane]) : T(0);
      const int nc = (int)min((unsigned)CC, c_hi - c0);
      for (int cb = 0; cb < nc; cb += RE_D) {
#pragma unroll
        for (int t = 0; t < RE_D; ++t) {
          if (cb + t >= nc) break;
          cp_async_wait<RE_D - 1>();         // this column's copies (the oldest group) have landed
          T v[R], rec[R];
          lds_run<T, R>(ring + t * 32 * R, v);
          issue(t);                          // the slot refills with the column D ahead
          ub.times(hc + (cb + t) * RM, r1, rec);
          T s = T(0);
#pragma unroll
          for (int q = 0; q < R; ++q) {
            const T d = v[q] - rec[q];
            s = fma(wr[q] * d, d, s);
          }
          csum = fma(__shfl_sync(0xffffffffu, wl, cb + t), s, csum);
        }
        bad |= !isfinite(csum);
        acc += (double)csum;
        csum = T(0);
      }
    }
    cp_async_wait<0>();
  }
  acc = block_sum(acc, sh);
  if (bad && flags) atomicOr(flags, kFlagNonFinite);
  if (threadIdx.x == 0) {
    partial[blockIdx.x] = acc;
    __threadfence();
    last = (atomicAdd(counter, 1u) == gridDim.x - 1);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double t = 0.0;
  for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) t += __ldcg(&partial[b]);
  t = block_sum(t, sh);
  if (threadIdx.x == 0) {
    *out = t;
    atomicExch(counter, 0u);
  }
}

template <typename T>
void launch_recon_err(const T* V, const T* U1, const T* H, int r1, int N1, int64_t ncol, const T* w1, const T* wcol,
                      double* partial, unsigned* counter, int nblocks, double* out, unsigned* flags, cudaStream_t s,
                      const int* gate) {
  // rows per lane: 16 bytes of V (float ranks above 16: 8 bytes), so that U_1 stays in registers
  const uintptr_t va = (uintptr_t)V;
  auto go = [&](auto kern, auto rows, auto rmax) {
    constexpr int R = decltype(rows)::value, RM = decltype(rmax)::value;
    // two CTAs per SM at most, and at least a ring of columns for every warp (a small tensor's
    // warps would spend their time on U_1, and a batch's members on each other's SMs)
    const int64_t units = ((N1 + 32 * R - 1) / (32 * R)) * ncol;
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>({(units + 8 * RE_D - 1) / (8 * RE_D), nblocks, 2 * 152}));
    const size_t sm = sizeof(T) * 8 * (RE_D * 32 * R + 2 * kChunk<T, RM> * RM);
    if (sm > 47 * 1024) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    const int vec = N1 % R == 0 && va % (R * sizeof(T)) == 0;
    kern<<<blocks, 256, sm, s>>>(V, U1, H, r1, N1, (unsigned)ncol, w1, wcol, vec, partial, counter, out, flags, gate);
    count_launch();
  };
  if constexpr (sizeof(T) == 4) {
    if (r1 <= 8) go(k_recon_err_rows<float, 4, 8>, IntC<4>(), IntC<8>());
    else if (r1 <= 12) go(k_recon_err_rows<float, 4, 12>, IntC<4>(), IntC<12>());
    else if (r1 <= 16) go(k_recon_err_rows<float, 4, 16>, IntC<4>(), IntC<16>());
    else go(k_recon_err_rows<float, 2, 32>, IntC<2>(), IntC<32>());
  } else {
    if (r1 <= 8) go(k_recon_err_rows<double, 2, 8>, IntC<2>(), IntC<8>());
    else if (r1 <= 16) go(k_recon_err_rows<double, 2, 16>, IntC<2>(), IntC<16>());
    else go(k_recon_err_rows<double, 1, 32>, IntC<1>(), IntC<32>());
  }
}
template void launch_recon_err<float>(const float*, const float*, const float*, int, int, int64_t, const float*,
                                      const float*, double*, unsigned*, int, double*, unsigned*, cudaStream_t,
                                      const int*);
template void launch_recon_err<double>(const double*, const double*, const double*, int, int, int64_t, const double*,
                                       const double*, double*, unsigned*, int, double*, unsigned*, cudaStream_t,
                                       const int*);

// Weights in the compute type: w_1 (N_1) and the column weights of the mode-1 unfolding,
// w_c = prod_{m>1} w_m(i_m) for c = i_2 + N_2 (i_3 + ...).
template <typename T>
__global__ void k_weights_T(WeightView wv, T* __restrict__ w1, T* __restrict__ wcol) {
  const unsigned N1 = (unsigned)wv.N[0];
  unsigned ncol = 1;
  for (int m = 1; m < wv.p; ++m) ncol *= (unsigned)wv.N[m];
  for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < N1 + ncol; e += gridDim.x * blockDim.x) {
    if (e < N1) {
      w1[e] = (T)wv.w[0][e];
    } else {
      unsigned rem = e - N1;
      double wc = 1.0;
      for (int m = 1; m < wv.p; ++m) {
        const unsigned nm = (unsigned)wv.N[m];
        wc *= wv.w[m][rem % nm];
        rem /= nm;
      }
      wcol[e - N1] = (T)wc;
    }
  }
}

template <typename T>
void launch_weights_T(const WeightView& wv, T* w1, T* wcol, cudaStream_t s) {
  k_weights_T<T><<<152, 256, 0, s>>>(wv, w1, wcol);
  count_launch();
}
template void launch_weights_T<float>(const WeightView&, float*, float*, cudaStream_t);
template void launch_weights_T<double>(const WeightView&, double*, double*, cudaStream_t);

// ---------------------------------------------------------------------------
// Generic n-mode product
// ---------------------------------------------------------------------------

// K large, L == 1: one warp per output column q, lanes split k, JT accumulators.
template <typename Tin, typename Tm, typename Tacc, int JT>
__global__ void k_mp_reduce_col(const Tin* __restrict__ in, Tacc* __restrict__ out, const Tm* __restrict__ M, int K,
                                int J, int64_t Q, int64_t sMj, int64_t sMk) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t q = warp; q < Q; q += nwarps) {
    const Tin* col = in + q * K;
    for (int j0 = 0; j0 < J; j0 += JT) {
      Tacc acc[JT];
#pragma unroll
      for (int t = 0; t < JT; ++t) acc[t] = Tacc(0);
      for (int k = lane; k < K; k += 32) {
        Tacc v = (Tacc)col[k];
#pragma unroll
        for (int t = 0; t < JT; ++t)
          if (j0 + t < J) acc[t] += (Tacc)M[(j0 + t) * sMj + k * sMk] * v;
      }
#pragma unroll
      for (int t = 0; t < JT; ++t) {
        Tacc v = warp_sum(acc[t]);
        if (lane == 0 && j0 + t < J) out[(j0 + t) + (int64_t)J * q] = v;
      }
    }
  }
}

// K large, Q == 1, J <= 32: out (L x J) = in (L x K) M^T as a tiled product.  A CTA
// owns 64 consecutive l and all j; K in chunks of 32 staged in shared memory (in along
// l: coalesced; M once per chunk), the next chunk loaded into registers while the
// current one is multiplied; thread (tl, tj) accumulates l = 4 tl .. 4 tl + 3 and
// j = 2 tj, 2 tj + 1.  Fixed summation order over k.
template <typename Tin, typename Tm, typename Tacc>
__global__ void __launch_bounds__(256) k_mp_gemm(const Tin* __restrict__ in, Tacc* __restrict__ out,
                                                 const Tm* __restrict__ M, int64_t L, int K, int J, int64_t sMj,
                                                 int64_t sMk) {
  constexpr int BM = 64, BK = 32;
  __shared__ Tacc As[BK][BM + 1];
  __shared__ Tacc Bs[BK][33];
  const int tid = threadIdx.x;
  const int tl = tid & 15, tj = tid >> 4;
  for (int64_t l0 = blockIdx.x * (int64_t)BM; l0 < L; l0 += (int64_t)gridDim.x * BM) {
    Tacc acc[4][2];
#pragma unroll
    for (int x = 0; x < 4; ++x) acc[x][0] = acc[x][1] = Tacc(0);
    // register staging of one chunk: 8 entries of in, 4 of M per thread
    Tacc ra[8], rb[4];
    auto fetch = [&](int k0) {
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int e = tid + 256 * u, i = e % BM, kk = e / BM;
        const int64_t l = l0 + i;
        const int k = k0 + kk;
        ra[u] = (l < L && k < K) ? (Tacc)in[l + L * (int64_t)k] : Tacc(0);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = tid + 256 * u, j = e % 32, kk = e / 32;
        const int k = k0 + kk;
        rb[u] = (j < J && k < K) ? (Tacc)M[j * sMj + (int64_t)k * sMk] : Tacc(0);
      }
    };
    fetch(0);
    for (int k0 = 0; k0 < K; k0 += BK) {
      __syncthreads();
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int e = tid + 256 * u;
        As[e / BM][e % BM] = ra[u];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = tid + 256 * u;
        Bs[e / 32][e % 32] = rb[u];
      }
      __syncthreads();
      if (k0 + BK < K) fetch(k0 + BK);
#pragma unroll 8
      for (int kk = 0; kk < BK; ++kk) {
        Tacc a[4], b[2];
#pragma unroll
        for (int x = 0; x < 4; ++x) a[x] = As[kk][4 * tl + x];
        b[0] = Bs[kk][2 * tj];
        b[1] = Bs[kk][2 * tj + 1];
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          acc[x][0] = fma(a[x], b[0], acc[x][0]);
          acc[x][1] = fma(a[x], b[1], acc[x][1]);
        }
      }
    }
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = 0; y < 2; ++y) {
        const int64_t l = l0 + 4 * tl + x;
        const int j = 2 * tj + y;
        if (l < L && j < J) out[l + L * (int64_t)j] = acc[x][y];
      }
  }
}

// K large, L > 1: one thread per (l, q), l fastest (coalesced over l).
template <typename Tin, typename Tm, typename Tacc, int JT>
__global__ void k_mp_reduce_gen(const Tin* __restrict__ in, Tacc* __restrict__ out, const Tm* __restrict__ M,
                                int64_t L, int K, int J, int64_t Q, int64_t sMj, int64_t sMk) {
  const unsigned total = (unsigned)(L * Q), uL = (unsigned)L;
  for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    const unsigned l = e % uL, q = e / uL;
    const Tin* base = in + l + (size_t)uL * K * q;
    for (int j0 = 0; j0 < J; j0 += JT) {
      Tacc acc[JT];
#pragma unroll
      for (int t = 0; t < JT; ++t) acc[t] = Tacc(0);
      for (int k = 0; k < K; ++k) {
        Tacc v = (Tacc)base[(int64_t)k * L];
#pragma unroll
        for (int t = 0; t < JT; ++t)
          if (j0 + t < J) acc[t] += (Tacc)M[(j0 + t) * sMj + k * sMk] * v;
      }
#pragma unroll
      for (int t = 0; t < JT; ++t)
        if (j0 + t < J) out[l + L * ((j0 + t) + (int64_t)J * q)] = acc[t];
    }
  }
}

// K large, L * Q small: one warp per (l, q), lanes split k, JT accumulators.
template <typename Tin, typename Tm, typename Tacc, int JT>
__global__ void k_mp_reduce_warp(const Tin* __restrict__ in, Tacc* __restrict__ out, const Tm* __restrict__ M,
                                 int64_t L, int K, int J, int64_t Q, int64_t sMj, int64_t sMk) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const unsigned uL = (unsigned)L;
  for (int64_t w = warp; w < L * Q; w += nwarps) {
    const unsigned l = (unsigned)w % uL, q = (unsigned)w / uL;
    const Tin* base = in + l + (size_t)uL * K * q;
    for (int j0 = 0; j0 < J; j0 += JT) {
      Tacc acc[JT];
#pragma unroll
      for (int t = 0; t < JT; ++t) acc[t] = Tacc(0);
      for (int k = lane; k < K; k += 32) {
        Tacc v = (Tacc)base[(int64_t)k * L];
#pragma unroll
        for (int t = 0; t < JT; ++t)
          if (j0 + t < J) acc[t] += (Tacc)M[(j0 + t) * sMj + k * sMk] * v;
      }
#pragma unroll
      for (int t = 0; t < JT; ++t) {
        Tacc v = warp_sum(acc[t]);
        if (lane == 0 && j0 + t < J) out[l + L * ((j0 + t) + (int64_t)J * q)] = v;
      }
    }
  }
}

// K large, very few (l, q): one block per (l, q), threads split k, block reduction.
template <typename Tin, typename Tm, typename Tacc, int JT>
__global__ void k_mp_reduce_block(const Tin* __restrict__ in, Tacc* __restrict__ out, const Tm* __restrict__ M,
                                  int64_t L, int K, int J, int64_t Q, int64_t sMj, int64_t sMk) {
  __shared__ Tacc sh[JT][33];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const unsigned uL = (unsigned)L;
  for (unsigned w = blockIdx.x; w < (unsigned)(L * Q); w += gridDim.x) {
    const unsigned l = w % uL, q = w / uL;
    const Tin* base = in + l + (size_t)uL * K * q;
    for (int j0 = 0; j0 < J; j0 += JT) {
      Tacc acc[JT];
#pragma unroll
      for (int t = 0; t < JT; ++t) acc[t] = Tacc(0);
      for (int k = threadIdx.x; k < K; k += blockDim.x) {
        Tacc v = (Tacc)base[(size_t)k * uL];
#pragma unroll
        for (int t = 0; t < JT; ++t)
          if (j0 + t < J) acc[t] += (Tacc)M[(j0 + t) * sMj + k * sMk] * v;
      }
#pragma unroll
      for (int t = 0; t < JT; ++t) {
        Tacc v = warp_sum(acc[t]);
        if (lane == 0) sh[t][wid] = v;
      }
      __syncthreads();
      if (threadIdx.x < JT && j0 + (int)threadIdx.x < J) {
        Tacc v = Tacc(0);
        for (int x = 0; x < nw; ++x) v += sh[threadIdx.x][x];
        out[l + uL * ((j0 + threadIdx.x) + (size_t)J * q)] = v;
      }
      __syncthreads();
    }
  }
}

// K small: a thread per output element (l, j, q), l fastest.  For few outputs: bound by the
// latency of the K loads and of the chain of products, so eight terms' loads are in flight
// while the eight before are multiplied.
template <typename Tin, typename Tm, typename Tacc>
__global__ void k_mp_expand1(const Tin* __restrict__ in, Tacc* __restrict__ out, const Tm* __restrict__ M, int64_t L,
                             int K, int J, int64_t Q, int64_t sMj, int64_t sMk, const int* __restrict__ gate) {
  if (gate && *gate == 0) return;
  const unsigned total = (unsigned)(L * J * Q), uL = (unsigned)L, uJ = (unsigned)J;
  for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    const unsigned l = e % uL;
    const unsigned jq = e / uL;
    const unsigned j = jq % uJ;
    const unsigned q = jq / uJ;
    const Tin* base = in + l + (size_t)uL * K * q;
    const Tm* mrow = M + j * sMj;
    // eight terms at a time, the next eight's loads issued before the current products
    Tacc acc = Tacc(0), a[8], b[8];
    auto fetch = [&](int k) {
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        a[t] = k + t < K ? (Tacc)__ldg(&mrow[(k + t) * sMk]) : Tacc(0);
        b[t] = k + t < K ? (Tacc)__ldg(&base[(size_t)(k + t) * uL]) : Tacc(0);
      }
    };
    fetch(0);
    for (int k = 0; k < K; k += 8) {
      Tacc x[8], y[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) { x[t] = a[t]; y[t] = b[t]; }
      if (k + 8 < K) fetch(k + 8);
#pragma unroll
      for (int t = 0; t < 8; ++t)
        if (k + t < K) acc = fma(x[t], y[t], acc);
    }
    out[e] = acc;
  }
}

// K small, many outputs: a thread per output element, l fastest, K products in order.  Where the
// lanes of a thread per (l, q) would be empty (a last mode far longer than the product of the
// others' ranks and sizes), and for double outputs that are no fewer than their inputs: double runs at its
// arithmetic, which the finest grain shares out best (reconstructions of 7 x 100 000 at rank 7 17 us
// against 62 with eight outputs a thread, 126^3 at rank 14 65 against 72; float 7 x 100 000 12 against 25).
template <typename Tin, typename Tm, typename Tacc>
__global__ void __launch_bounds__(256) k_mp_expand_out(const Tin* __restrict__ in, Tacc* __restrict__ out,
                                                       const Tm* __restrict__ M, int64_t L, int K, int J, int64_t Q,
                                                       int64_t sMj, int64_t sMk, const int* __restrict__ gate) {
  if (gate && *gate == 0) return;
  const unsigned total = (unsigned)(L * J * Q), uL = (unsigned)L, uJ = (unsigned)J;
  for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    const unsigned l = e % uL, jq = e / uL, j = jq % uJ, q = jq / uJ;
    const Tin* base = in + l + (size_t)uL * K * q;
    const Tm* mrow = M + j * sMj;
    Tacc acc = Tacc(0);
    for (int k = 0; k < K; ++k) acc = fma((Tacc)__ldg(&mrow[k * sMk]), (Tacc)base[(size_t)k * uL], acc);
    out[e] = acc;
  }
}

// K small: a thread per (l, q), l fastest, and JT consecutive outputs j: every value of `in` is
// read once for the JT of them, their M (blockIdx.y's rows) comes from shared memory.  Each
// output sums its K products in order whatever JT is.  Bound: the stores of L J Q values;
// r_1 N_2 N_3 = 11 x 128 x 512 from K = 16: 5.6 us, where a thread per output (K reads of both
// operands for each) took 9.7 us.  Taken where that makes two CTAs per SM and half of the last
// JT are not wasted.
template <typename Tin, typename Tm, typename Tacc, int JT>
__global__ void __launch_bounds__(256) k_mp_expand(const Tin* __restrict__ in, Tacc* __restrict__ out,
                                                   const Tm* __restrict__ M, int64_t L, int K, int J, int64_t Q,
                                                   int64_t sMj, int64_t sMk, const int* __restrict__ gate) {
  if (gate && *gate == 0) return;
  __shared__ Tacc Ms[64 * JT];                       // [k][jj]
  const unsigned total = (unsigned)(L * Q), uL = (unsigned)L, uJ = (unsigned)J;
  for (int j0 = blockIdx.y * JT; j0 < J; j0 += gridDim.y * JT) {
    __syncthreads();
    for (int e = threadIdx.x; e < K * JT; e += blockDim.x) {
      const int k = e / JT, j = j0 + e % JT;
      Ms[e] = j < J ? (Tacc)M[j * sMj + k * sMk] : Tacc(0);
    }
    __syncthreads();
    for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
      const unsigned l = e % uL, q = e / uL;
      const Tin* base = in + l + (size_t)uL * K * q;
      Tacc acc[JT];
#pragma unroll
      for (int t = 0; t < JT; ++t) acc[t] = Tacc(0);
#pragma unroll 4
      for (int k = 0; k < K; ++k) {
        const Tacc v = (Tacc)base[(size_t)k * uL];
#pragma unroll
        for (int t = 0; t < JT; ++t) acc[t] = fma(Ms[k * JT + t], v, acc[t]);
      }
      Tacc* o = out + l + (size_t)uL * (j0 + (size_t)uJ * q);
#pragma unroll
      for (int t = 0; t < JT; ++t)
        if (j0 + t < J) o[(size_t)t * uL] = acc[t];
    }
  }
}

// Float, L == 1, K large: out[j + J q] = sum_k M[j, k] in[k + K q], the first contraction of a
// (re)initialisation's core (V x_1 A_1^T).  A warp takes eight columns q at a time, its lanes
// four k of each 128; four outputs at a time are summed over the lanes by a transposing
// butterfly (lane l ends with column l % 8, output l / 8).  M in shared memory, zero past K.
// Bound: HBM (K Q values read once); 256 x 128 x 512 at 11 outputs: 33 us, where a warp per
// column with M from global memory took 160 us.
__global__ void __launch_bounds__(256) k_mp_cols(const float* __restrict__ in, float* __restrict__ out,
                                                 const float* __restrict__ M, int K, int J, unsigned Q, int64_t sMj,
                                                 int64_t sMk, int vec) {
  extern __shared__ __align__(16) float mc_sm[];       // [J rounded up to 4][Kp]
  const int Kp = (K + 127) & ~127, Jp = (J + 3) & ~3;
  for (int e = threadIdx.x; e < Jp * Kp; e += blockDim.x) {
    const int j = e / Kp, k = e % Kp;
    mc_sm[e] = (j < J && k < K) ? M[j * sMj + k * sMk] : 0.f;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const unsigned nw = gridDim.x * (blockDim.x >> 5);
  for (unsigned g = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); g * 8 < Q; g += nw) {
    const unsigned q0 = g * 8;
    for (int j0 = 0; j0 < Jp; j0 += 16) {              // sixteen outputs in registers at a time
      float acc[4][32];
#pragma unroll
      for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int i = 0; i < 32; ++i) acc[b][i] = 0.f;
      for (int k0 = 0; k0 < Kp; k0 += 128) {
        const int k = k0 + 4 * lane;
        float4 v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          v[c] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (q0 + c < Q) {
            const float* src = in + (size_t)K * (q0 + c) + k;
            if (vec) {
              if (k < K) v[c] = __ldg((const float4*)src);
            } else {
              if (k < K) v[c].x = __ldg(src);
              if (k + 1 < K) v[c].y = __ldg(src + 1);
              if (k + 2 < K) v[c].z = __ldg(src + 2);
              if (k + 3 < K) v[c].w = __ldg(src + 3);
            }
          }
        }
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          if (j0 + 4 * b >= Jp) break;
#pragma unroll
          for (int a = 0; a < 4; ++a) {
            const float4 m = *(const float4*)&mc_sm[(j0 + 4 * b + a) * Kp + k];
#pragma unroll
            for (int c = 0; c < 8; ++c)
              acc[b][c + 8 * a] = fmaf(v[c].w, m.w, fmaf(v[c].z, m.z, fmaf(v[c].y, m.y, fmaf(v[c].x, m.x, acc[b][c + 8 * a]))));
          }
        }
      }
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        if (j0 + 4 * b >= Jp) break;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const bool up = lane & o;
#pragma unroll
          for (int i = 0; i < o; ++i) {
            const float keep = up ? acc[b][i + o] : acc[b][i], send = up ? acc[b][i] : acc[b][i + o];
            acc[b][i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
          }
        }
        const unsigned q = q0 + (lane & 7);
        const int j = j0 + 4 * b + (lane >> 3);
        if (q < Q && j < J) out[j + (size_t)J * q] = acc[b][0];
      }
    }
  }
}

// V^TDB = U_1 H in float with H = T x_2 U_2 ... x_p U_p (r_1 x ncol): the last and only large product of
// a reconstruction.  Lane l of a warp owns R rows of a block of 32 R with U_1's in registers
// and walks a range of columns, 32 columns' H at a time in shared memory (padded to RM, zeros past
// r_1), the next 32 on their way by cp.async.  Bound: HBM, N_1 ncol values written once.
// 256 x 128 x 512 float at r_1 = 11, 17.7 us from a cold cache (18.3 with H through registers);
// a whole reconstruction of 192 x 129 x 192 x 3 at r_1 = 13 31.7 us (33.0), where the product
// of the last mode with a thread per output took 91 us, and the mode before it as long.  A warp
// takes eight columns at least: 64^3 float at rank 4 in 11 us, with 32 at least 15 us.
template <int R, int RM>
__global__ void __launch_bounds__(256, 2) k_recon_out(const float* __restrict__ U1, const float* __restrict__ H, int r1,
                                                      int N1, unsigned ncol, int vec, float* __restrict__ V) {
  using T = float;
  constexpr int CC = kChunk<T, RM>;
  extern __shared__ __align__(16) unsigned char ro_raw[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  T* hs = (T*)ro_raw + (size_t)wib * 2 * CC * RM;       // two chunks of H
  for (int e = lane; e < 2 * CC * RM; e += 32) hs[e] = T(0);
  const int nrb = (N1 + 32 * R - 1) / (32 * R);
  const unsigned gw = blockIdx.x * (blockDim.x >> 5) + wib, tw = gridDim.x * (blockDim.x >> 5);
  const unsigned wpr = tw >= (unsigned)nrb ? tw / nrb : 1u;
  const unsigned kk = gw % wpr;
  const unsigned c_lo = (unsigned)((uint64_t)ncol * kk / wpr), c_hi = (unsigned)((uint64_t)ncol * (kk + 1) / wpr);
  for (unsigned rb = gw / wpr; rb < (unsigned)nrb && c_lo < c_hi; rb += (tw >= (unsigned)nrb ? (unsigned)nrb : tw)) {
    const int i0 = (int)rb * 32 * R + R * lane;
    __syncwarp();                            // hs cleared, and the row block before is done with it
    fetch_columns<T, RM>(hs, H, r1, c_lo, c_hi, lane);
    cp_async_commit();
    RowBlock<T, R, RM> ub;
    ub.load(U1, i0, N1, r1);
    int par = 0;                             // the half of hs that holds this chunk
    for (unsigned c0 = c_lo; c0 < c_hi; c0 += CC, par ^= 1) {
      cp_async_wait<0>();
      __syncwarp();
      fetch_columns<T, RM>(hs + CC * RM * (par ^ 1), H, r1, c0 + CC, c_hi, lane);
      cp_async_commit();
      const T* hc = hs + CC * RM * par;
      const int nc = (int)min((unsigned)CC, c_hi - c0);
      for (int c = 0; c < nc; ++c) {
        T rec[R];
        ub.times(hc + c * RM, r1, rec);
        T* o = V + (size_t)N1 * (c0 + c) + i0;
        if (vec) {
          if (i0 < N1) {
            if constexpr (R == 4)
              __stcs((float4*)o, make_float4(rec[0], rec[1], rec[2], rec[3]));
            else
              __stcs((float2*)o, make_float2(rec[0], rec[1]));
          }
        } else {
#pragma unroll
          for (int q = 0; q < R; ++q)
            if (i0 + q < N1) __stcs(o + q, rec[q]);
        }
      }
    }
    cp_async_wait<0>();
  }
}

// Mode 1 last where its rows fill a warp's lanes and the last mode does not; the mode products in
// order elsewhere.  Float, us of a reconstruction, this against the products: 7 x 100 000 (rank 4)
// 31 to 11, 24 x 200 x 200 (4) 15 to 12, 33 x 300 x 300 (14) 29 to 21, 64 x 3 x 64 x 64 (4) 30 to 20,
// 130 x 300 x 300 (4) 27 to 25; 80 x 120 x 120 (4) 12 to 13, 260 x 300 x 300 (4) 33 to 39, 192 x 129 x
// 192 x 3 (14) 37 to 74; two modes 10 to 8.  The lines: three fifths of the rows that a warp's blocks
// hold, or a quarter beside a last mode that is next to uncompressed.  Double runs at its arithmetic,
// which the products share out better: 64^3 (4) 17 to 14, 130 x 300 x 300 (4) 242 to 93, 300 x 200 x 3
// (12) 30 to 17; at 256 x 128 x 64 (14) 72 us each, at 192 x 129 x 192 x 3 (14) 427 to 451.
bool recon_mode1_last(int p, const int64_t* N, const int* r) {
  if (p == 2) return false;
  const bool short_last = 4 * (int64_t)r[p - 1] >= 3 * N[p - 1];
  return 5 * N[0] >= 3 * 128 * ((N[0] + 127) / 128) || (N[0] >= 32 && short_last);
}

void launch_recon_out(const float* U1, const float* H, int r1, int N1, int64_t ncol, float* V, cudaStream_t s) {
  using T = float;
  const uintptr_t va = (uintptr_t)V;
  auto go = [&](auto kern, auto rows, auto rmax) {
    constexpr int R = decltype(rows)::value, RM = decltype(rmax)::value;
    const size_t sm = sizeof(T) * 8 * 2 * kChunk<T, RM> * RM;
    if (sm > 48 * 1024) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    // a warp per eight columns of a row block at least, two CTAs per SM at most
    const int64_t units = ((N1 + 32 * R - 1) / (32 * R)) * ((ncol + 7) / 8);
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((units + 7) / 8, 2 * 152));
    const int vec = N1 % R == 0 && va % (R * sizeof(T)) == 0;
    kern<<<blocks, 256, sm, s>>>(U1, H, r1, N1, (unsigned)ncol, vec, V);
    count_launch();
  };
  if (r1 <= 8) go(k_recon_out<4, 8>, IntC<4>(), IntC<8>());
  else if (r1 <= 12) go(k_recon_out<4, 12>, IntC<4>(), IntC<12>());
  else if (r1 <= 16) go(k_recon_out<4, 16>, IntC<4>(), IntC<16>());
  else go(k_recon_out<2, 32>, IntC<2>(), IntC<32>());
}

// H = T x_2 U_2 x_3 U_3 (x_4 U_4) in float, r_1 x N_2 x slices, in one launch: a CTA forms the
// r_1 x r_2 slice G = sum_j T[:, :, j] c_j, c_j = U_3[i_3, c] U_4[i_4, d] over the J = r_3 r_4
// pairs, then its block of columns G U_2[i_2, :]^T.  Bound: latency; 256 x 128 x 512 at (11, 8,
// 16) 8.2 us against 9.1 in two mode products with the gap between them.
constexpr int CC_T = 256, CC_JMAX = 1024, CC_NB = 256, CC_PRE = 16;
struct CoreCols {
  const float* T;
  const float* U2;
  const float* U3;
  const float* U4;               // null: three modes
  float* H;
  int r1, r2, r3, J, N2, N3, N4, nb;         // nb: columns i_2 of a CTA
};
__global__ void __launch_bounds__(CC_T) k_core_cols(CoreCols a, const int* __restrict__ gate) {
  if (gate && *gate == 0) return;
  extern __shared__ __align__(16) float cc_sm[];
  const int r12 = a.r1 * a.r2, neg = (r12 + 31) >> 5;       // groups of 32 entries of G
  float* cj = cc_sm;                                       // J
  float* G = cj + a.J;                                     // r12
  float* U2s = G + r12;                                    // r2 x nb
  float* red = U2s + a.r2 * a.nb;                          // groups of j x 32 neg
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int s = blockIdx.x, i3 = s % a.N3, i4 = s / a.N3;
  const int lo = blockIdx.y * a.nb, nc = min(a.nb, a.N2 - lo);
  for (int j = t; j < a.J; j += CC_T) {
    const float c = __ldg(&a.U3[i3 + a.N3 * (j % a.r3)]);
    cj[j] = a.U4 ? c * __ldg(&a.U4[i4 + a.N4 * (j / a.r3)]) : c;
  }
  for (int b = w; b < a.r2; b += CC_T / 32)
    for (int il = lane; il < a.nb; il += 32) U2s[il + a.nb * b] = il < nc ? __ldg(&a.U2[lo + il + a.N2 * b]) : 0.f;
  // the eight warps over the groups of entries and, where these are few, over runs of j; the
  // first CC_PRE values of T are on their way before the wait for c_j
  const int js = max(1, (CC_T / 32) / neg), nq = neg * js;
  float pre[CC_PRE];
  {
    const int e = 32 * (w % neg) + lane, jlo = a.J * (w / neg) / js, jhi = a.J * (w / neg + 1) / js;
#pragma unroll
    for (int u = 0; u < CC_PRE; ++u)
      pre[u] = (w < nq && e < r12 && jlo + u < jhi) ? __ldg(&a.T[e + (size_t)r12 * (jlo + u)]) : 0.f;
  }
  __syncthreads();
  for (int q = w; q < nq; q += CC_T / 32) {
    const int eg = q % neg, jg = q / neg, e = 32 * eg + lane;
    const int jlo = a.J * jg / js, jhi = a.J * (jg + 1) / js;
    const float* src = a.T + (e < r12 ? e : 0);
    float g = 0.f;
    int j = jlo;
    if (q == w) {
#pragma unroll
      for (int u = 0; u < CC_PRE; ++u)
        if (jlo + u < jhi) g = fmaf(pre[u], cj[jlo + u], g);
      j = min(jhi, jlo + CC_PRE);
    }
#pragma unroll 8
    for (; j < jhi; ++j) g = fmaf(__ldg(&src[(size_t)r12 * j]), cj[j], g);
    if (js > 1) red[jg * 32 * neg + e] = g;
    else if (e < r12) G[e] = g;
  }
  __syncthreads();
  if (js > 1) {
    if (t < r12) {
      float g = red[t];
      for (int jg = 1; jg < js; ++jg) g += red[jg * 32 * neg + t];
      G[t] = g;
    }
    __syncthreads();
  }
  // output a1 + r1 il, a1 and il carried from one to the next
  float* out = a.H + (size_t)a.r1 * (lo + (size_t)a.N2 * s);
  const int dil = CC_T / a.r1, da = CC_T - dil * a.r1;
  int il = t / a.r1, a1 = t - il * a.r1;
  for (int e = t; e < a.r1 * nc; e += CC_T) {
    float h = 0.f;
#pragma unroll 8
    for (int b = 0; b < a.r2; ++b) h = fmaf(G[a1 + a.r1 * b], U2s[il + a.nb * b], h);
    out[e] = h;
    il += dil;
    a1 += da;
    if (a1 >= a.r1) { a1 -= a.r1; ++il; }
  }
}

// Three and four modes, where forming G again for every slice and column block costs less than
// the launch it saves (2^24 multiply-adds, 2 us); false: not taken.
bool launch_core_cols(const float* T, const float* const* U, int p, const int64_t* N, const int* r, float* H,
                      cudaStream_t s, const int* gate) {
  if (p < 3 || p > 4) return false;
  CoreCols a;
  a.T = T;
  a.U2 = U[1];
  a.U3 = U[2];
  a.U4 = p == 4 ? U[3] : nullptr;
  a.H = H;
  a.r1 = r[0];
  a.r2 = r[1];
  a.r3 = r[2];
  a.J = r[2] * (p == 4 ? r[3] : 1);
  a.N2 = (int)N[1];
  a.N3 = (int)N[2];
  a.N4 = p == 4 ? (int)N[3] : 1;
  const int64_t ns = (int64_t)a.N3 * a.N4;
  // columns of a CTA: two CTAs per SM where the slices alone are fewer, 16 columns at least
  const int64_t sub = std::max<int64_t>((a.N2 + CC_NB - 1) / CC_NB, std::min<int64_t>((2 * 152 + ns - 1) / ns, (a.N2 + 15) / 16));
  a.nb = (int)((a.N2 + sub - 1) / sub);
  const int64_t ny = (a.N2 + a.nb - 1) / a.nb;
  const int r12 = a.r1 * a.r2, neg = (r12 + 31) / 32;
  if (a.J > CC_JMAX || ny > 65535 || (int64_t)r12 * a.J * ns * ny > (1 << 24)) return false;
  const size_t sm = sizeof(float) * (a.J + r12 + (size_t)a.r2 * a.nb + 32 * std::max(8, neg));
  if (sm > 48 * 1024) return false;
  k_core_cols<<<dim3((unsigned)ns, (unsigned)ny), CC_T, sm, s>>>(a, gate);
  count_launch();
  return true;
}

template <typename Tin, typename Tm, typename Tacc>
void launch_modeprod(const Tin* in, Tacc* out, const Tm* M, int64_t L, int K, int J, int64_t Q, int64_t sMj,
                     int64_t sMk, cudaStream_t s, const int* gate) {
  if (L <= 0 || K <= 0 || J <= 0 || Q <= 0) return;
  count_launch();
  if (K <= 64) {
    const int64_t lq = L * Q;
    if ((lq < 128 || (sizeof(Tacc) == 8 && J >= K)) && lq * J >= 2 * 152 * 256) {
      k_mp_expand_out<Tin, Tm, Tacc><<<(unsigned)std::min<int64_t>((lq * J + 255) / 256, 152 * 32), 256, 0, s>>>(
          in, out, M, L, K, J, Q, sMj, sMk, gate);
    } else if (J >= 5 && ((lq + 255) / 256) * ((J + 7) / 8) >= 2 * 152) {
      const dim3 grid((unsigned)std::min<int64_t>((lq + 255) / 256, 152 * 32), (unsigned)std::min((J + 7) / 8, 16384));
      k_mp_expand<Tin, Tm, Tacc, 8><<<grid, 256, 0, s>>>(in, out, M, L, K, J, Q, sMj, sMk, gate);
    } else if (((lq + 255) / 256) * ((J + 3) / 4) >= 2 * 152) {
      const dim3 grid((unsigned)std::min<int64_t>((lq + 255) / 256, 152 * 32), (unsigned)std::min((J + 3) / 4, 16384));
      k_mp_expand<Tin, Tm, Tacc, 4><<<grid, 256, 0, s>>>(in, out, M, L, K, J, Q, sMj, sMk, gate);
    } else {
      // blocks small enough to reach every SM (double issues 64 cycles apart on each)
      const int64_t total = lq * J;
      int block = 256;
      while (block > 64 && (total + block - 1) / block < 2 * 152) block /= 2;
      k_mp_expand1<Tin, Tm, Tacc><<<(unsigned)std::min<int64_t>((total + block - 1) / block, 152 * 32), block, 0, s>>>(
          in, out, M, L, K, J, Q, sMj, sMk, gate);
    }
    return;
  }
  if constexpr (std::is_same<Tin, float>::value && std::is_same<Tm, float>::value && std::is_same<Tacc, float>::value) {
    const size_t sm = (size_t)((J + 3) & ~3) * ((K + 127) & ~127) * sizeof(float);
    if (L == 1 && Q >= 1024 && sm <= 160 * 1024) {
      if (sm > 48 * 1024) cudaFuncSetAttribute(k_mp_cols, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
      const int vec = (K & 3) == 0 && ((uintptr_t)in & 15) == 0;
      const int blocks = (int)std::min<int64_t>((Q + 63) / 64, 152);
      k_mp_cols<<<blocks, 256, sm, s>>>(in, out, M, K, J, (unsigned)Q, sMj, sMk, vec);
      return;
    }
    // few rows: a block per (l, q) splits K, where 64-row tiles would leave most SMs idle
    // (88 x 512 by 16: 7.5 against 29 us with two CTAs)
    if (Q == 1 && L > 1 && L <= 256) {
      const int blocks = (int)std::min<int64_t>(L, 152 * 8);
      if (J <= 8) k_mp_reduce_block<Tin, Tm, Tacc, 8><<<blocks, 256, 0, s>>>(in, out, M, L, K, J, Q, sMj, sMk);
      else if (J <= 16) k_mp_reduce_block<Tin, Tm, Tacc, 16><<<blocks, 256, 0, s>>>(in, out, M, L, K, J, Q, sMj, sMk);
      else k_mp_reduce_block<Tin, Tm, Tacc, 32><<<blocks, 256, 0, s>>>(in, out, M, L, K, J, Q, sMj, sMk);
      return;
    }
  }
  if (Q == 1 && L >= 64 && J <= 32) {
    const int blocks = (int)std::min<int64_t>((L + 63) / 64, 152 * 8);
    k_mp_gemm<Tin, Tm, Tacc><<<blocks, 256, 0, s>>>(in, out, M, L, K, J, sMj, sMk);
  } else if (L > 1 && L * Q <= 1024) {
    int blocks = (int)std::min<int64_t>(L * Q, 152 * 8);
    if (J <= 8)
      k_mp_reduce_block<Tin, Tm, Tacc, 8><<<blocks, 256, 0, s>>>(in, out, M, L, K, J, Q, sMj, sMk);
    else if (J <= 16)
      k_mp_reduce_block<Tin, Tm, Tacc, 16><<<blocks, 256, 0, s>>>(in, out, M, L, K, J, Q, sMj, sMk);
    else
      k_mp_reduce_block<Tin, Tm, Tacc, 32><<<blocks, 256, 0, s>>>(in, out, M, L, K, J, Q, sMj, sMk);
  } else if (L > 1 && L * Q <= 32768) {
    int64_t warps = L * Q;
    int blocks = (int)std::min<int64_t>((warps * 32 + 255) / 256, 152 * 32);
    if (J <= 8)
      k_mp_reduce_warp<Tin, Tm, Tacc, 8><<<blocks, 256, 0, s>>>(in, out, M, L, K, J, Q, sMj, sMk);
    else if (J <= 16)
      k_mp_reduce_warp<Tin, Tm, Tacc, 16><<<blocks, 256, 0, s>>>(in, out, M, L, K, J, Q, sMj, sMk);
    else
      k_mp_reduce_warp<Tin, Tm, Tacc, 32><<<blocks, 256, 0, s>>>(in, out, M, L, K, J, Q, sMj, sMk);
  } else if (L == 1) {
    int64_t warps = Q;
    int blocks = (int)std::min<int64_t>((warps * 32 + 255) / 256, 152 * 32);
    if (J <= 8)
      k_mp_reduce_col<Tin, Tm, Tacc, 8><<<blocks, 256, 0, s>>>(in, out, M, K, J, Q, sMj, sMk);
    else if (J <= 16)
      k_mp_reduce_col<Tin, Tm, Tacc, 16><<<blocks, 256, 0, s>>>(in, out, M, K, J, Q, sMj, sMk);
    else
      k_mp_reduce_col<Tin, Tm, Tacc, 32><<<blocks, 256, 0, s>>>(in, out, M, K, J, Q, sMj, sMk);
  } else {
    int64_t total = L * Q;
    int blocks = (int)std::min<int64_t>((total + 127) / 128, 152 * 32);
    if (J <= 8)
      k_mp_reduce_gen<Tin, Tm, Tacc, 8><<<blocks, 128, 0, s>>>(in, out, M, L, K, J, Q, sMj, sMk);
    else if (J <= 16)
      k_mp_reduce_gen<Tin, Tm, Tacc, 16><<<blocks, 128, 0, s>>>(in, out, M, L, K, J, Q, sMj, sMk);
    else
      k_mp_reduce_gen<Tin, Tm, Tacc, 32><<<blocks, 128, 0, s>>>(in, out, M, L, K, J, Q, sMj, sMk);
  }
}

#define INST_MP(Tin, Tm, Tacc)                                                                                   \
  template void launch_modeprod<Tin, Tm, Tacc>(const Tin*, Tacc*, const Tm*, int64_t, int, int, int64_t, int64_t, \
                                               int64_t, cudaStream_t, const int*);
INST_MP(float, float, float)
INST_MP(double, double, double)

}  // namespace tdb
