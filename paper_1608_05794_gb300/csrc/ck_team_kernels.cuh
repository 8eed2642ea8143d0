// Device code and launch helpers shared by the team-per-reactor kernels
// (one CTA per reactor): shared-memory carving, the reactor work queue, the
// forward-difference Jacobian, the error norm and the starting step of the
// integrators, and the occupancy-sized persistent grid.
#pragma once
#include <cuda_runtime.h>

#include "ck_internal.h"
#include "ck_team.cuh"

namespace ck {

// Next reactor index for this CTA from the global queue (same in every thread).
static __device__ __forceinline__ int team_next(int32_t* queue, int* slot) {
  if (threadIdx.x == 0) *slot = atomicAdd(queue, 1);
  team_sync();
  const int r = *slot;
  team_sync();
  return r;
}

// Forward-difference Jacobian (the paper's choice for ROS4, Sec. 5), with
// the increments of CVODE's dense difference quotients: unit roundoff U,
// weights w_i = 1/(atol + rtol |y_i|), fnorm = WRMS_w(f(y)), floor
// s0 = 1000 |h| U n fnorm (1 when fnorm = 0), and column j =
// (f(y + s_j e_j) - f(y)) / s_j with s_j = max(sqrt(U) |y_j|, s0 / w_j).
// f0 = f(y) is computed here (unless have_f0: the caller already holds it
// for this y) and reused as the first stage's f; the n columns cost n team
// RHS evaluations.  y_o, f0_o, yt_o, f_o: offsets of n-vectors in shared
// memory (the last two scratch); bufs_o, vp, qq as in team_rhs.
template <bool INT, bool LAT = false>
static __device__ __noinline__ void team_jacobian_fd(const DevMech& d, const double* tab, double p, int y_o, double h,
                                                     double rtol, double atol, int f0_o, double* J, int ldj, int yt_o,
                                                     int f_o, int bufs_o, int vp, RhsQ qq, bool have_f0 = false) {
  extern __shared__ __align__(16) double sm[];
  const double* y = sm + y_o;
  const double* f0 = sm + f0_o;
  const double* F = sm + f_o;
  double* Yt = sm + yt_o;
  const int n = d.n, tid = (int)threadIdx.x;
  if (!have_f0) team_rhs_any<INT, false, LAT>(d, tab, p, y_o, f0_o, bufs_o, vp, qq);
  double s = 0.0;
  if (tid < vp)
    for (int i = tid; i < n; i += vp) {
      const double v = f0[i] / (atol + rtol * fabs(y[i]));
      s = fma(v, v, s);
      Yt[i] = y[i];
    }
  const double fn = sqrt(team_sum(s, sm + bufs_o) / n);
  const double U = 2.220446049250313080847e-16;  // 2^-52
  const double srur = 1.490116119384765625e-8;   // 2^-26 = sqrt(U)
  const double s0 = (fn != 0.0) ? 1000.0 * fabs(h) * U * n * fn : 1.0;
  for (int j = 0; j < n; ++j) {
    const double sj = fmax(srur * fabs(y[j]), s0 * (atol + rtol * fabs(y[j])));
    if (tid == 0) Yt[j] = y[j] + sj;
    team_sync();
    team_rhs_any<INT, false, LAT>(d, tab, p, yt_o, f_o, bufs_o, vp, qq);
    for (int i = tid; i < n; i += blockDim.x) J[(size_t)i * ldj + j] = (F[i] - f0[i]) / sj;
    if (tid == 0) Yt[j] = y[j];
    team_sync();
  }
}

// x^q, the step-size controller's power, by the first warp alone and handed
// to the others through red[SC_POW]: pow is long, and every warp that runs it
// pays all of its FP64 instructions.  x is the same in every thread; every
// thread must call it.
static __device__ __forceinline__ double team_pow(double x, double q, double* red) {
  if (blockDim.x == 32) return pow(x, q);
  if (threadIdx.x == 0) red[SC_POW] = pow(x, q);
  __syncthreads();
  return red[SC_POW];
}

// Weighted RMS norm over the team (reading shared with the oracle:
// sqrt(mean (e_i / (atol + rtol max(|y_i|, |ynew_i|)))^2)).  vp: the lanes
// that the components are dealt to (as the species sums).  ORD: the components
// one after another (the sum by every thread).
template <bool ORD = false>
static __device__ __forceinline__ double team_wrms(int n, double* e, const double* y0, const double* y1,
                                                   double rtol, double atol, double* red, int vp) {
  const int tid = threadIdx.x;
  double s = 0.0;
  if (tid < vp)
    for (int i = tid; i < n; i += vp) {
      const double sc = atol + rtol * fmax(fabs(y0[i]), fabs(y1[i]));
      const double v = e[i] / sc;
      if (ORD) e[i] = v;
      else s = fma(v, v, s);
    }
  if (ORD) {
    team_sync();
    for (int i = 0; i < n; ++i) s = fma(e[i], e[i], s);
    team_sync();
  } else {
    s = team_sum(s, red);
  }
  return sqrt(s / n);
}

// Initial step, Hairer-Norsett-Wanner starting-step algorithm (order 4).
// Offsets, vp and qq as in team_rhs; f0, y1, f1 are scratch vectors.
template <bool INT, bool LAT = false>
static __device__ __noinline__ double team_h0(const DevMech& d, const double* tab, double p, int y0_o, double tspan,
                                              double rtol, double atol, int f0_o, int y1_o, int f1_o, int bufs_o,
                                              int vp, RhsQ qq) {
  extern __shared__ __align__(16) double sm[];
  const double *y0 = sm + y0_o, *f0 = sm + f0_o, *f1 = sm + f1_o;
  double *y1 = sm + y1_o, *red = sm + bufs_o;
  const int n = d.n, tid = (int)threadIdx.x;
  const bool lane_in = tid < vp;
  team_rhs_any<INT, false, LAT>(d, tab, p, y0_o, f0_o, bufs_o, vp, qq);
  double s0 = 0.0, s1 = 0.0;
  if (lane_in)
    for (int i = tid; i < n; i += vp) {
      const double sc = atol + rtol * fabs(y0[i]);
      s0 = fma(y0[i] / sc, y0[i] / sc, s0);
      s1 = fma(f0[i] / sc, f0[i] / sc, s1);
    }
  const double d0 = sqrt(team_sum(s0, red) / n);
  const double d1 = sqrt(team_sum(s1, red) / n);
  const double ha = (d0 < 1e-5 || d1 < 1e-5) ? 1e-6 : 0.01 * d0 / d1;
  for (int i = tid; i < n; i += blockDim.x) y1[i] = fma(ha, f0[i], y0[i]);
  team_sync();
  team_rhs_any<INT, false, LAT>(d, tab, p, y1_o, f1_o, bufs_o, vp, qq);
  double s2 = 0.0;
  if (lane_in)
    for (int i = tid; i < n; i += vp) {
      const double sc = atol + rtol * fabs(y0[i]);
      const double v = (f1[i] - f0[i]) / sc;
      s2 = fma(v, v, s2);
    }
  const double d2 = sqrt(team_sum(s2, red) / n) / ha;
  const double dm = fmax(d1, d2);
  const double hb = (dm <= 1e-15) ? fmax(1e-6, ha * 1e-3) : pow(0.01 / dm, 0.2);
  return fmin(fmin(100.0 * ha, hb), tspan);
}

// ------------------------------------------------------------------ launch helpers
// The mechanism for a kernel that keeps `fixed` doubles beside its rates of
// progress: with all of them at once where that leaves room for `ctas` CTAs an
// SM, else in the loader's chunks (the same sums in the same order).
static inline DevMech with_rates(const HostMech& hm, size_t fixed, int ctas) {
  DevMech d = hm.d;
  if (hm.R > 0) d.rhs_chunk = hm.R;
  if (fixed + rhs_doubles(d) > (size_t)smem_doubles(ctas)) d.rhs_chunk = hm.d.rhs_chunk;
  return d;
}

// Persistent grid: as many CTAs of `kernel` as fit on every SM (or the
// caller's cap), at most one per work item.
template <class K>
static inline int team_grid(K kernel, int threads, size_t smem, int64_t work, const LaunchCfg& cfg) {
  // the same limit in every call: another thread may be about to launch this
  // kernel with more
  if (smem > 48 * 1024)
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(double) * smem_doubles(1));
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
  if (per_sm < 1) per_sm = 1;
  if (cfg.ctas_per_sm > 0 && cfg.ctas_per_sm < per_sm) per_sm = cfg.ctas_per_sm;
  int64_t g = (int64_t)per_sm * sm_count();
  if (work < g) g = work;
  return (int)(g < 1 ? 1 : g);
}

}  // namespace ck
