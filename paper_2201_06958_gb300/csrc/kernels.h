// kernels.h - host-side launchers of libtdb's kernels (internal C++ interface).
#pragma once

#include <algorithm>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "common.cuh"

namespace tdb {

// Bump allocator over the caller's workspace (256-byte aligned pieces); with a
// null base it only measures.
struct Carver {
  char* base;
  size_t off = 0;
  explicit Carver(void* b) : base((char*)b) {}
  template <typename T>
  T* take(size_t count) {
    off = (off + 255) & ~(size_t)255;
    T* p = base ? (T*)(base + off) : nullptr;
    off += count * sizeof(T);
    return p;
  }
};


struct WeightView {
  int p;
  int64_t N[kMaxModes];
  const double* w[kMaxModes];
};

// The weighted Cholesky-QR of freshly computed bases (k_small.cu).
struct RowArgs {
  ModeDesc d;
  const double* w[kMaxModes];
  const double* Rinv;            // p x LD x LD
  double* Up[kMaxModes];
  double* Uout[kMaxModes];
  void* A[kMaxModes];            // weighted bases (Ta)
  double* part;                  // p x ntile x LD x LD
  int ntile;                     // tiles per mode in `part`
};

// Arguments of the fused per-step update (k_update.cu).  Tc is the compute type;
// r x r matrices are column-major with leading dimension kMaxRank.
struct UpdArgs {
  ModeDesc d;
  const void* Y[kMaxModes];      // projections Y_n (Tc)
  const void* dS;                // core increment (Tc)
  const void* ds_y2;             // Y_2 (Tc): when set, phase 1 forms dS = Y_2 x_2 A_2^T
  void* dS_out;                  // ... into this buffer (the one dS points to)
  double* T;                     // core (in: step k, out: step k+1)
  double* T2;                    // scratch core
  void* Tcore;                   // Tc copy of the core (in and out; aliases T in FP64)
  double* U[kMaxModes];          // bases (in and out)
  double* Up[kMaxModes];         // U' (scratch)
  void* X[kMaxModes];            // M G^{-1} (Tc scratch, N_n x r_n)
  const double* w[kMaxModes];    // quadrature weights
  void* A[kMaxModes];            // W U (Tc; in: step k, out: step k+1)
  void* Uc[kMaxModes];           // U (Tc; in and out)
  double* G;                     // p x LD x LD (out)
  double* Ginv;                  // p x LD x LD (out)
  float* Ginvf;                  // float copy of Ginv (in: of the core of step k; out), null in FP64
  double* R;                     // p x LD x LD (out)
  double* Rinv;                  // p x LD x LD (out)
  double* sig2;                  // p x LD, descending (out)
  float* Vprev;                  // p x LD x LD, eigenvectors of G_n (Jacobi warm start; in and out)
  void* part;                    // 2 x p x ntile x LD x LD partial sums (Tc scratch)
  void* red;                     // 2 x kMaxModes x LD x LD sums of the partials of modes over 1024 points (Tc)
  double* gpart;                 // p x gsplit x LD x LD Gram partials (scratch)
  int ntile, gsplit;
  int warm, reorth;
  int skip_finish;               // phase 7 (G, G^{-1}, sigma^2) left to launch_gram_finish
  // Heun's second stage: the right-hand side is evaluated at the predicted state held in
  // T/U, and the new state is (y_k + y_pred + increment) / 2 with y_k = (T0, U0_n) in
  // the layout of T/U.  Null for an Euler step (and for Heun's first stage).
  const double* T0;
  const double* U0[kMaxModes];
  int combine;                   // with T0: 1 = Heun's mean (T0 + T + dT) / 2, 2 = T0 + dT (midpoint)
  unsigned* bar;                 // arrival counter of the grid barriers (zero at the launch)
  unsigned long long* stamps;    // per-phase timer stamps (profiling), or null
  unsigned* flags;
};

struct GramView {
  int p, n;
  int64_t N[kMaxModes];
  const double* w[kMaxModes];
  int64_t L, Q, Nn;
};

// A timing event on stream s: an external event-record node while s is being captured
// (so that the replayed graph records it), an ordinary record otherwise.
inline cudaError_t record_timing_event(cudaEvent_t ev, cudaStream_t s) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs == cudaStreamCaptureStatusActive)
    return cudaEventRecordWithFlags(ev, s, cudaEventRecordExternal);
  return cudaEventRecord(ev, s);
}

// Process-wide count of libtdb kernel launches (tdb_kernel_launches).
void count_launch(int n = 1);
long long launches_so_far();

// k_basic.cu
struct StateViews {
  const double* src;             // the state to take, or null: T and U hold it
  double* T;
  double* U[kMaxModes];
  const double* w[kMaxModes];
  void* Tcore;                   // compute-type core (T itself in FP64)
  void* A[kMaxModes];
  void* Uc[kMaxModes];
  int64_t N[kMaxModes], nT, total;
  int r[kMaxModes];
  int bases;                     // form A_n too
};
template <typename T> void launch_state_views(const StateViews& v, cudaStream_t s);
void launch_state_pack(const StateViews& v, double* out, cudaStream_t s);
template <typename Ts, typename Td> void launch_cast(const Ts* a, Td* b, int64_t n, cudaStream_t s);
template <typename T>
void launch_diff_norm(const T* a, const T* b, T* out, int N1, int64_t ncol, T scale, const T* w1, const T* wcol,
                      const WeightView& wv,
                      double* partial, unsigned* counter, int nblocks, double* norm2, unsigned* flags, cudaStream_t s);
template <typename T>
void launch_recon_err(const T* V, const T* U1, const T* H, int r1, int N1, int64_t ncol, const T* w1, const T* wcol,
                      double* partial, unsigned* counter, int nblocks, double* out, unsigned* flags, cudaStream_t s,
                      const int* gate = nullptr);
// Whether a float reconstruction takes mode 1 last, in launch_recon_out
bool recon_mode1_last(int p, const int64_t* N, const int* r);
// V = U1 H (N1 x ncol; H: r1 x ncol)
void launch_recon_out(const float* U1, const float* H, int r1, int N1, int64_t ncol, float* V, cudaStream_t s);
// H = T x_2 U_2 ... x_p U_p in one launch (three and four modes of few enough products), or false
bool launch_core_cols(const float* T, const float* const* U, int p, const int64_t* N, const int* r, float* H,
                      cudaStream_t s, const int* gate);
template <typename T>
void launch_weights_T(const WeightView& wv, T* w1, T* wcol, cudaStream_t s);
template <typename Tin, typename Tm, typename Tacc>
void launch_modeprod(const Tin* in, Tacc* out, const Tm* M, int64_t L, int K, int J, int64_t Q, int64_t sMj,
                     int64_t sMk, cudaStream_t s, const int* gate = nullptr);

// Column slices of the Gram partials G_n = T_(n) T_(n)^T: one per 32 columns of the
// widest unfolding, at most `cap`.  The fused update and the standalone refresh use
// the same split, so both sum in the same order.
inline int gram_split(const int* r, int p, int cap) {
  int64_t Rprod = 1, maxcol = 1;
  for (int n = 0; n < p; ++n) Rprod *= r[n];
  for (int n = 0; n < p; ++n) maxcol = std::max<int64_t>(maxcol, Rprod / r[n]);
  return (int)std::min<int64_t>(cap, std::max<int64_t>(1, maxcol / 32));
}

// k_update.cu (standalone Gram refresh)
// Phase 7 of the update alone (p CTAs): G_n, G_n^{-1}, sigma^(n) from the Gram partials.
void launch_gram_finish(const ModeDesc& d, const double* Gpart, int nsplit, double* G, double* Ginv, float* Ginvf,
                        double* sig2, float* Vprev, int warm, unsigned* flags, cudaStream_t s);
void launch_gram(const ModeDesc& d, const double* T, double* Gpart, int nsplit, double* G, double* Ginv,
                 float* Ginvf, double* sig2, float* Vprev, int warm, unsigned* flags, cudaStream_t s);

// k_small.cu
template <typename Tc>
void launch_orthonormalize(RowArgs& a, double* R, double* Rinv, unsigned* flags, cudaStream_t s);

// CTAs that hold all of dS = Y_2 x_2 A_2^T at once (eight threads of 1024 per element)
__host__ __device__ inline int64_t update_ds_ctas(int64_t rprod) { return (rprod + 127) / 128; }

// Phases that a profiled update times: those of the kernel (k_update.cu), whatever the modes.
constexpr int kUpdPhases = 7;

// k_update.cu: a.bar must hold zero
template <typename Tc>
tdb_status launch_update(UpdArgs& a, int grid_hint, cudaStream_t s);

// The updates of n states of the float compute type, phase by phase over all of them:
// part 0 = phases 1-6, part 1 = phase 7 (G_n, G_n^{-1}, sigma^(n)).
constexpr int kUpdBatch = 16;
void launch_update_batch(const UpdArgs* args, int n, int part, cudaStream_t s);

// k_eig.cu (float compute types)
void launch_sqrt_weights(const double* w, int n, float* ws, cudaStream_t s);
void launch_weight_data(const float* V, int p, const int64_t* N, const float* const* ws, int64_t S, float* Vw,
                        cudaStream_t s);
// Vw Vw^T of a mode of Nn points (L, Q: the sizes before and after it) into C64; part:
// gram_part_elems(Nn, L Q) doubles.
size_t gram_part_elems(int64_t Nn, int64_t ncol);
void launch_gram_weighted(const float* Vw, int64_t L, int64_t Nn, int64_t Q, double* part, double* C64,
                          cudaStream_t s);

// k_eig_modes.cu: leading eigenpairs of several symmetric positive semi-definite matrices
constexpr int kEigBlock = 50;              // most columns of a block: 16 more than the wanted pairs (<= 34)
constexpr int kEigSweeps = 32;             // Jacobi sweeps at most
constexpr int kEigWhole = 96;              // most points of a mode that can be solved whole
constexpr int kEigPart = 3840;             // a group's sums: block^2 and its upper triangle, and 64
struct EigProblem {
  const double* C;                         // n x n, symmetric
  int n, k;                                // k wanted pairs, k <= min(n, 34)
  double* scratch;                         // eig_modes_scratch(n, k) doubles
  double* ev;                              // k eigenvalues, descending
  double* Q;                               // n x k eigenvectors, entry of largest magnitude positive
  double* trace;
};
struct EigMode {
  const double* C;
  int n, m, k, mp;                         // m columns of the block, mp: padded to eight
  int cta0, nct;                           // the CTAs of the group
  double* Q;                               // n x m block, row-major (ld mp)
  double* part;                            // per-CTA partial sums (stride pstride), and column statistics
  int pstride;
  double* sums;                            // the group's sums
  double* rot;                             // Jacobi rotations, by sweep, round and pair
  unsigned* bar;                           // group barrier
  unsigned* done;                          // Jacobi sweeps done
  double* ev;
  double* out;
  double* trace;
  double tau, least;
};
struct EigModes {
  int p;
  EigMode mode[kMaxModes];
  unsigned* flags;
};
size_t eig_modes_scratch(int n, int k);
// All p problems in one cooperative launch.  tau: relative accuracy of the matrices' entries
// (what the iteration converges to); least: pairs below it, relative to the largest, are waited
// for three rounds at most.
tdb_status launch_eig_modes(EigProblem* pr, int p, double tau, double least, unsigned* flags, cudaStream_t s);

// k_hosvd.cu
template <typename Tv>
void launch_wgram(const Tv* V, const GramView& g, double* part, size_t part_cap, double* C64, cudaStream_t s);
void launch_scale_basis(const double* Q, const double* w, int64_t n, int r, double* U, cudaStream_t s);
void launch_merge_weights(const WeightView& wv, int skip, int64_t M, double* wq, cudaStream_t s);
template <typename Tv>
void launch_short_map(const Tv* V, int first, int64_t Nn, int64_t M, const double* wn, const double* sqw,
                      const double* Z, const double* ev, int k, double* Q, cudaStream_t s);

}  // namespace tdb
