// Team-per-reactor kernels: analytic and forward-difference Jacobians,
// batched dense LU / solve and RKF45 with one CTA per reactor, and the
// dispatch of the ROS4 integrator (its kernels live in ck_ros4_*.cu).  CTAs
// pull reactors from a global atomic counter (dynamic scheduling,
// granularity one reactor).
#include <cuda_runtime.h>

#include <mutex>

#include "ck_team_kernels.cuh"

namespace ck {

// ------------------------------------------------------------------ RHS (team)
// The sums are in the order of k_rhs, and the bits the same.
template <bool INT>
__global__ void __launch_bounds__(128) k_rhs_team(const __grid_constant__ DevMech d, int64_t N,
                                                  const double* __restrict__ p, const double* __restrict__ y,
                                                  double* __restrict__ f) {
  extern __shared__ __align__(16) double sm[];
  const int n = d.n;
  const RhsQ qq{2 * n + species_doubles(d.S), d.rhs_chunk};
  for (int64_t r = blockIdx.x; r < N; r += gridDim.x) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) sm[i] = y[r * n + i];
    team_sync();
    team_rhs_any<INT, false, !INT>(d, d.tab, p[r], 0, n, 2 * n, 256, qq);
    for (int i = threadIdx.x; i < n; i += blockDim.x) f[r * n + i] = sm[n + i];
  }
}

// ------------------------------------------------------------------ Jacobian
// The matrix is assembled in place in the output (its lines stay in L2), so
// that a CTA's shared memory holds the per-reaction values instead.
template <int P, int MINB>
__global__ void __launch_bounds__(P, MINB) k_jacobian(const __grid_constant__ DevMech d, int64_t N,
                                                  const double* __restrict__ p, const double* __restrict__ y,
                                                  double* __restrict__ jac) {
  extern __shared__ __align__(16) double sm[];
  const int n = d.n;
  double* ys = sm + d.wide.scratch;
  double* fs = ys + n;
  for (int64_t r = blockIdx.x; r < N; r += gridDim.x) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) ys[i] = y[r * n + i];
    team_sync();
    team_jacobian<(P > 64)>(d, d.wide, d.tab, p[r], ys, fs, jac + r * (int64_t)n * n, nullptr, 0,
                  carve_bufs(fs + n, d.S, sm, d.wide.chunk, 256));
  }
}

// Forward-difference Jacobians (one CTA per reactor), as ROS4 builds them
// with the forward-difference option at step size h[r].  INT: products in integer
// arithmetic (111 species: 150 reactors 2.40 ms against 3.05).
template <bool INT>
__global__ void __launch_bounds__(256) k_jacobian_fd(const __grid_constant__ DevMech d, int64_t N,
                                                     const double* __restrict__ p, const double* __restrict__ y,
                                                     const double* __restrict__ h, double rtol, double atol,
                                                     double* __restrict__ jac) {
  extern __shared__ __align__(16) double sm[];
  const int n = d.n, ys = n * n;
  const RhsQ qq{ys + 4 * n + species_doubles(d.S), d.rhs_chunk};
  for (int64_t r = blockIdx.x; r < N; r += gridDim.x) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) sm[ys + i] = y[r * n + i];
    team_sync();
    team_jacobian_fd<INT>(d, d.tab, p[r], ys, h[r], rtol, atol, ys + n, sm, n, ys + 2 * n, ys + 3 * n, ys + 4 * n,
                          n > 64 ? 256 : 64, qq);
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) jac[r * (int64_t)n * n + e] = sm[e];
    team_sync();
  }
}

// ------------------------------------------------------------------ batched LU
// A dim x dim matrix into shared memory, rows ld apart, eight loads a thread
// in flight.
static __device__ __forceinline__ void load_matrix(double* A, int ld, const double* __restrict__ src, int dim, float rc) {
  const int nn = dim * dim, P = blockDim.x;
  for (int e0 = threadIdx.x; e0 < nn; e0 += 8 * P) {
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = e0 + u * P < nn ? src[e0 + u * P] : 0.0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int e = e0 + u * P;
      if (e < nn) A[e + flat_row(e, rc) * (ld - dim)] = v[u];
    }
  }
}

// Shared memory, in doubles: the matrix, 1 / U_kk, the row tables and pivots.
static __host__ __device__ __forceinline__ size_t lu_doubles(int dim) {
  return (((size_t)dim * lu_ld(dim) + 1) & ~(size_t)1) + 4 * (size_t)dim + 2 * (size_t)dim;
}
__global__ void __launch_bounds__(256) k_lu_factor(int64_t batch, int dim, double* __restrict__ a,
                                                   int32_t* __restrict__ piv, int32_t* __restrict__ info) {
  extern __shared__ __align__(16) double sm[];
  __shared__ int flag[2];
  const int nn = dim * dim, ld = lu_ld(dim), lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  double* A = sm;
  LuRow<double>* lr = reinterpret_cast<LuRow<double>*>(A + ((dim * lu_ld(dim) + 1) & ~1));
  double* invd = reinterpret_cast<double*>(lr + 2 * dim);
  int* rof = reinterpret_cast<int*>(invd + dim);
  int* pv = rof + dim;
  const float rc = 1.0f / (float)dim;
  for (int64_t m = blockIdx.x; m < batch; m += gridDim.x) {
    double* am = a + m * nn;
    load_matrix(A, ld, am, dim, rc);
    team_sync();
    const int inf = lu_flat<false>(A, dim, rof, pv, invd, lr, flag);
    for (int i = warp; i < dim; i += nw) {
      const double* row = A + (rof[i] >> 8);
      for (int j = lane; j < dim; j += 32) am[i * dim + j] = row[j];
    }
    for (int i = threadIdx.x; i < dim; i += blockDim.x) piv[m * dim + i] = pv[i];
    if (threadIdx.x == 0) info[m] = inf;
    team_sync();
  }
}

__global__ void k_lu_solve(int64_t batch, int dim, const double* __restrict__ lu,
                           const int32_t* __restrict__ piv, double* __restrict__ bvec) {
  extern __shared__ __align__(16) double sm[];
  const int nn = dim * dim, ld = lu_ld(dim);
  double* A = sm;
  double* invd = A + (dim - 1) * ld + dim;
  int* pv = reinterpret_cast<int*>(invd + dim);
  double* x = invd + dim + (dim + 1) / 2;
  const float rc = 1.0f / (float)dim;
  for (int64_t m = blockIdx.x; m < batch; m += gridDim.x) {
    load_matrix(A, ld, lu + m * nn, dim, rc);
    for (int i = threadIdx.x; i < dim; i += blockDim.x) {
      pv[i] = piv[m * dim + i];
      x[i] = bvec[m * dim + i];
    }
    team_sync();
    for (int i = threadIdx.x; i < dim; i += blockDim.x) invd[i] = rcp_rn(A[i * ld + i]);
    team_sync();
    if (threadIdx.x < 32) warp_lu_solve(A, dim, pv, invd, x);
    team_sync();
    for (int i = threadIdx.x; i < dim; i += blockDim.x) bvec[m * dim + i] = x[i];
    team_sync();
  }
}

// ------------------------------------------------------------------ RKF45 (team)
// RKF45 with one CTA per reactor (the paper's "deep" form): the six stage
// right-hand sides are evaluated by the team, so a reactor's working set
// (8 n-vectors, the species arrays and the rates of progress) stays in shared
// memory and the number of steps of one reactor never holds back another.
// Bound by the FP64 unit (87 % active, 608 warp instructions a right-hand side
// of the 53-species mechanism before the integer products): 16384 reactors 266
// ms, 362 with 710 instructions.
//
// TAIL: reactors that the thread-per-reactor kernel handed on (the entries of
// list, *count of them but cap at most), taken up where it left them; every sum
// is then in that kernel's order, so that its results do not depend on where
// a reactor is finished.
template <bool INT, bool TAIL>
static __device__ __forceinline__ void rkf45_team(const DevMech& d, int64_t N, const double* __restrict__ p,
                                                  double* __restrict__ y, const double* __restrict__ dt,
                                                  double* h_io, const SolverParams& sp, int32_t* steps,
                                                  int32_t* status, int32_t* queue, const RkCont* list) {
  extern __shared__ __align__(16) double sm[];
  __shared__ int slot;
  const int n = d.n;
  double* yv = sm;
  double* yt = yv + n;
  double* kk = yt + n;  // six stages, n each
  constexpr int vp = 64;
  const int o_y = 0, o_t = n, o_k = 2 * n, bufs = 8 * n;
  double* red = sm + bufs;
  const RhsQ qq{bufs + species_doubles(d.S), d.rhs_chunk};
  const bool fixed = sp.fixed_h > 0.0;
  const int tid = (int)threadIdx.x, P = blockDim.x;
  double* k0 = kk;
  double* k1 = kk + n;
  double* k2 = kk + 2 * n;
  double* k3 = kk + 3 * n;
  double* k4 = kk + 4 * n;
  double* k5 = kk + 5 * n;
  for (;;) {
    int r = team_next(queue, &slot);
    if (r >= N) break;
    RkCont from{};
    if (TAIL) {
      from = list[r];
      r = from.r;
    }
    for (int i = tid; i < n; i += P) yv[i] = y[(int64_t)r * n + i];
    const double pr = p[r];
    const double tf = dt[r];
    team_sync();
    int bad = 0;
    for (int i = tid; i < n; i += P) bad |= !isfinite(yv[i]);
    bad = __syncthreads_or(bad);
    bad |= !(pr > 0.0) || !isfinite(pr) || !(yv[0] > 0.0) || !isfinite(tf) || !(tf >= 0.0);
    int st = ST_OK, acc = from.acc, rej = from.rej;
    double h = 0.0;
    if (!TAIL && bad) {
      st = ST_BADINPUT;
    } else if (tf > 0.0) {
      if (TAIL) h = from.h;
      else if (fixed) h = sp.fixed_h;
      else if (h_io && h_io[r] > 0.0) h = h_io[r];
      else if (sp.h0 > 0.0) h = sp.h0;
      else h = team_h0<INT, !INT>(d, d.tab, pr, o_y, tf, sp.rtol, sp.atol, o_k, o_t, o_k + n, bufs, vp, qq);
      const double hmin = 1e-15 * tf;
      double t = from.t;
      bool last_rej = from.last_rej != 0, last_nf = from.last_nf != 0;
      while (t < tf) {
        if (acc + rej >= sp.max_steps) { st = ST_MAXSTEPS; break; }
        const bool clamped = h >= tf - t;
        const double hh = clamped ? tf - t : h;
        if (hh < hmin) { st = last_nf ? ST_NONFINITE : ST_HMIN; break; }
        // k_s = hh f(y + sum_j a_sj k_j)
        team_rhs_any<INT, TAIL, !INT>(d, d.tab, pr, o_y, o_k, bufs, vp, qq);
        for (int i = tid; i < n; i += P) {
          k0[i] *= hh;
          yt[i] = fma(RK_A21, k0[i], yv[i]);
        }
        team_sync();
        team_rhs_any<INT, TAIL, !INT>(d, d.tab, pr, o_t, o_k + 1 * n, bufs, vp, qq);
        for (int i = tid; i < n; i += P) {
          k1[i] *= hh;
          yt[i] = fma(RK_A32, k1[i], fma(RK_A31, k0[i], yv[i]));
        }
        team_sync();
        team_rhs_any<INT, TAIL, !INT>(d, d.tab, pr, o_t, o_k + 2 * n, bufs, vp, qq);
        for (int i = tid; i < n; i += P) {
          k2[i] *= hh;
          yt[i] = fma(RK_A43, k2[i], fma(RK_A42, k1[i], fma(RK_A41, k0[i], yv[i])));
        }
        team_sync();
        team_rhs_any<INT, TAIL, !INT>(d, d.tab, pr, o_t, o_k + 3 * n, bufs, vp, qq);
        for (int i = tid; i < n; i += P) {
          k3[i] *= hh;
          yt[i] = fma(RK_A54, k3[i], fma(RK_A53, k2[i], fma(RK_A52, k1[i], fma(RK_A51, k0[i], yv[i]))));
        }
        team_sync();
        team_rhs_any<INT, TAIL, !INT>(d, d.tab, pr, o_t, o_k + 4 * n, bufs, vp, qq);
        for (int i = tid; i < n; i += P) {
          k4[i] *= hh;
          yt[i] = fma(RK_A65, k4[i],
                      fma(RK_A64, k3[i], fma(RK_A63, k2[i], fma(RK_A62, k1[i], fma(RK_A61, k0[i], yv[i])))));
        }
        team_sync();
        team_rhs_any<INT, TAIL, !INT>(d, d.tab, pr, o_t, o_k + 5 * n, bufs, vp, qq);
        // y* = y + sum b k (into yt), e = sum (bh - b) k (into k1, whose weights are 0)
        int nf = 0;
        for (int i = tid; i < n; i += P) {
          k5[i] *= hh;
          const double yn =
              fma(RK_B5, k4[i], fma(RK_B4, k3[i], fma(RK_B3, k2[i], fma(RK_B1, k0[i], yv[i]))));
          k1[i] = fma(RK_D6, k5[i], fma(RK_D5, k4[i], fma(RK_D4, k3[i], fma(RK_D3, k2[i], RK_D1 * k0[i]))));
          yt[i] = yn;
          nf |= !isfinite(yn);
        }
        nf = __syncthreads_or(nf);
        if (fixed) {
          for (int i = tid; i < n; i += P) yv[i] = yt[i];
          team_sync();
          t = clamped ? tf : t + hh;
          ++acc;
          continue;
        }
        const double e = team_wrms<TAIL>(n, k1, yv, yt, sp.rtol, sp.atol, red, vp);
        if (nf || !isfinite(e)) {
          ++rej;
          h = FAC_MIN * hh;
          last_rej = true;
          last_nf = true;
          continue;
        }
        last_nf = false;
        const double pe = (e == 0.0) ? 0.0 : team_pow(e, -0.2, red);
        if (e < 1.0) {
          for (int i = tid; i < n; i += P) yv[i] = yt[i];
          team_sync();
          t = clamped ? tf : t + hh;
          ++acc;
          double fac = (e == 0.0) ? FAC_MAX : fmin(FAC_MAX, fmax(FAC_MIN, SAFETY * pe));
          if (last_rej) fac = fmin(1.0, fac);
          h = hh * fac;
          last_rej = false;
        } else {
          ++rej;
          h = hh * fmax(FAC_MIN, SAFETY * pe);
          last_rej = true;
        }
      }
    }
    __syncthreads();
    for (int i = tid; i < n; i += P) y[(int64_t)r * n + i] = yv[i];
    if (tid == 0) {
      if (h_io && st != ST_BADINPUT && tf > 0.0) h_io[r] = h;
      if (steps) {
        steps[2 * (int64_t)r] = acc;
        steps[2 * (int64_t)r + 1] = rej;
      }
      status[r] = st;
    }
    __syncthreads();
  }
}

constexpr int RKF45_LAT_CTAS = 5;  // CTAs an SM of the latency form, by registers
template <bool INT>
__global__ void __launch_bounds__(128, INT ? 8 : RKF45_LAT_CTAS) k_rkf45_team(const __grid_constant__ DevMech d, int64_t N,
                                                       const double* __restrict__ p, double* __restrict__ y,
                                                       const double* __restrict__ dt, double* h_io, SolverParams sp,
                                                       int32_t* steps, int32_t* status, int32_t* queue) {
  rkf45_team<INT, false>(d, N, p, y, dt, h_io, sp, steps, status, queue, nullptr);
}

__global__ void __launch_bounds__(128, RKF45_LAT_CTAS) k_rkf45_tail(const __grid_constant__ DevMech d,
                                                       const double* __restrict__ p, double* __restrict__ y,
                                                       const double* __restrict__ dt, double* h_io, SolverParams sp,
                                                       int32_t* steps, int32_t* status, int32_t* queue,
                                                       const RkCont* __restrict__ list,
                                                       const int32_t* __restrict__ count, int cap) {
  const int n = *count < cap ? *count : cap;
  rkf45_team<false, true>(d, n, p, y, dt, h_io, sp, steps, status, queue, list);
}

// ------------------------------------------------------------------ launchers
cudaError_t launch_rhs_team(const HostMech& hm, int64_t n, const double* p, const double* y, double* f,
                            cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const size_t fixed = 2 * (size_t)hm.d.n + species_doubles(hm.S);
  const DevMech d = with_rates(hm, fixed, 4);
  const size_t smem = sizeof(double) * (fixed + rhs_doubles(d));
  const int threads = hm.S > 32 && hm.S <= 64 ? 96 : 128;
  LaunchCfg cfg;
  auto kern = hm.S > 32 ? k_rhs_team<true> : k_rhs_team<false>;
  const int grid = team_grid(kern, threads, smem, n, cfg);
  kern<<<grid, threads, smem, st>>>(d, n, p, y, f);
  return cudaGetLastError();
}

cudaError_t launch_jacobian(const HostMech& hm, int64_t n, const double* p, const double* y,
                            double* jac, cudaStream_t st, const LaunchCfg& cfg) {
  if (n <= 0) return cudaSuccess;
  const int nn = hm.d.n;
  const size_t smem =
      sizeof(double) * ((size_t)hm.d.wide.scratch + 2 * nn + species_doubles(hm.S) + 3 * hm.S);
  auto kern = nn <= 24 ? k_jacobian<64, 12> : (nn <= 64 ? k_jacobian<128, 6> : k_jacobian<256, 2>);
  const int threads = nn <= 24 ? 64 : (nn <= 64 ? 128 : 256);
  const int grid = team_grid(kern, threads, smem, n, cfg);
  kern<<<grid, threads, smem, st>>>(hm.d, n, p, y, jac);
  return cudaGetLastError();
}

cudaError_t launch_jacobian_fd(const HostMech& hm, int64_t n, const double* p, const double* y, const double* h,
                               double rtol, double atol, double* jac, cudaStream_t st, const LaunchCfg& cfg) {
  if (n <= 0) return cudaSuccess;
  const int nn = hm.d.n;
  const size_t fixed = (size_t)nn * nn + 4 * nn + species_doubles(hm.S);
  const DevMech d = with_rates(hm, fixed, n <= sm_count() ? 1 : team_ctas(nn));
  const size_t smem = sizeof(double) * (fixed + rhs_doubles(d));
  const int threads = nn <= 24 ? 64 : (nn <= 64 ? 96 : 256);
  auto kern = nn > 64 ? k_jacobian_fd<true> : k_jacobian_fd<false>;
  const int grid = team_grid(kern, threads, smem, n, cfg);
  kern<<<grid, threads, smem, st>>>(d, n, p, y, h, rtol, atol, jac);
  return cudaGetLastError();
}

cudaError_t launch_lu_factor(int64_t batch, int dim, double* a, int32_t* piv, int32_t* info,
                             cudaStream_t st) {
  if (batch <= 0) return cudaSuccess;
  LaunchCfg cfg;
  const size_t smem = sizeof(double) * lu_doubles(dim);
  // a warp alone needs no barriers and is enough for the smallest matrices,
  // except in a batch that leaves the SMs room (24: 300 matrices 40 us with one
  // warp, 32 with two; 1200 42 / 36; 2400 52 / 54); measured for 4096 matrices of
  // 54: 96 threads 712 us, 128 680
  const int threads = dim <= 24 ? (batch <= 8 * (int64_t)sm_count() ? 64 : 32) : (dim <= 64 ? 128 : 256);
  const int grid = team_grid(k_lu_factor, threads, smem, batch, cfg);
  k_lu_factor<<<grid, threads, smem, st>>>(batch, dim, a, piv, info);
  return cudaGetLastError();
}

cudaError_t launch_lu_solve(int64_t batch, int dim, const double* lu, const int32_t* piv,
                            double* b, cudaStream_t st) {
  if (batch <= 0) return cudaSuccess;
  const size_t smem = sizeof(double) * ((size_t)(dim - 1) * lu_ld(dim) + 3 * dim + (dim + 1) / 2);
  LaunchCfg cfg;
  // one warp solves, all load: as many as leave the residency to shared memory
  // (32: 4096 systems 35 us with 64 threads, 39 with 128; 54: 81 / 76)
  const int threads = dim <= 24 ? 32 : (dim <= 40 ? 64 : 128);
  const int grid = team_grid(k_lu_solve, threads, smem, batch, cfg);
  k_lu_solve<<<grid, threads, smem, st>>>(batch, dim, lu, piv, b);
  return cudaGetLastError();
}

size_t ros4_scratch_bytes_max() {
  static size_t cached[NOALLOC_MAX_DEVICES] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NOALLOC_MAX_DEVICES) return 0;
  if (!cached[dev]) {
    int smem_sm = 0;
    cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    // grid * (n^2 + n) * 8 <= grid * (shared memory of a CTA) <= SMs * (shared memory of an SM)
    cached[dev] = (size_t)sm_count() * (size_t)smem_sm;
  }
  return cached[dev];
}


constexpr int64_t ROS4_LAT_PER_SM = 4;
cudaError_t launch_ros4(const HostMech& hm, int64_t n, const double* p, double* y, const double* dt,
                        double* h_io, const SolverParams& sp, int32_t* steps, int32_t* status,
                        int32_t* queue, cudaStream_t st, const LaunchCfg& cfg, double* scratch,
                        size_t scratch_bytes, bool may_alloc) {
  if (n <= 0) return cudaSuccess;
  const int nn = hm.d.n;
  cudaError_t e = cudaMemsetAsync(queue, 0, sizeof(int32_t), st);
  if (e != cudaSuccess) return e;
  // Team sizes as measured on GB300.  10 species: two warps 234 / 343 ms on 512
  // / 4000 reactors, the latency form on four 205 / 454 (four of its teams
  // fit an SM: for batches they hold), one warp 272 / 375.  53 species, 4096
  // reactors: four warps 600 ms, two 731, three 667, six 646, eight 1031.  111
  // species, 1500 reactors: eight warps and two CTAs an SM 280 ms, twelve and
  // one 380.
  const bool lat = hm.S <= 32 && n <= ROS4_LAT_PER_SM * sm_count();
  auto* fn = cfg.grid_side == 16 ? launch_ros4_w8
             : nn <= 24          ? (lat ? launch_ros4_w4_lat : launch_ros4_w2)
                                 : (nn <= 64 ? launch_ros4_w4 : launch_ros4_w8);
  return fn(hm, n, p, y, dt, h_io, sp, steps, status, queue, st, cfg, scratch, scratch_bytes, may_alloc);
}

// Shared memory of a team RKF45 beside its rates, in doubles: eight vectors and
// the species arrays.
static size_t rkf45_fixed(const HostMech& hm) { return 8 * (size_t)hm.d.n + species_doubles(hm.S); }

cudaError_t launch_rkf45_team(const HostMech& hm, int64_t n, const double* p, double* y,
                              const double* dt, double* h_io, const SolverParams& sp, int32_t* steps,
                              int32_t* status, int32_t* queue, cudaStream_t st, const LaunchCfg& cfg) {
  if (n <= 0) return cudaSuccess;
  const int nn = hm.d.n;
  const size_t fixed = rkf45_fixed(hm);
  const DevMech d = with_rates(hm, fixed, hm.S > 32 ? 8 : RKF45_LAT_CTAS);
  const size_t smem = sizeof(double) * (fixed + rhs_doubles(d));
  // four warps shorten a step while the batch, or the caller's cap, leaves the
  // SMs room; two keep their lanes busier where neither does (53 species, four /
  // two warps: 300 reactors 13.0 / 19.0 ms, 1000 23.4 / 26.5, 2000 41.5 / 39.1,
  // 16384 278 / 268; 2000 capped at three CTAs an SM 18.3 / 23.1)
  const bool room = n < (int64_t)12 * sm_count() || (cfg.ctas_per_sm > 0 && cfg.ctas_per_sm < 12);
  const int threads = nn > 64 || hm.S <= 32 || room ? 128 : 64;
  auto kern = hm.S > 32 ? k_rkf45_team<true> : k_rkf45_team<false>;
  const int grid = team_grid(kern, threads, smem, n, cfg);
  cudaError_t e = cudaMemsetAsync(queue, 0, sizeof(int32_t), st);
  if (e != cudaSuccess) return e;
  kern<<<grid, threads, smem, st>>>(d, n, p, y, dt, h_io, sp, steps, status, queue);
  return cudaGetLastError();
}

bool rkf45_tail_takes(const HostMech& hm) {
  return with_rates(hm, rkf45_fixed(hm), RKF45_LAT_CTAS).rhs_chunk >= hm.R;
}

cudaError_t launch_rkf45_tail(const HostMech& hm, const double* p, double* y, const double* dt, double* h_io,
                              const SolverParams& sp, int32_t* steps, int32_t* status, int32_t* queue,
                              const RkCont* list, const int32_t* count, int cap, cudaStream_t st,
                              const LaunchCfg& cfg) {
  const size_t fixed = rkf45_fixed(hm);
  const DevMech d = with_rates(hm, fixed, RKF45_LAT_CTAS);
  const size_t smem = sizeof(double) * (fixed + rhs_doubles(d));
  const int threads = 128;
  const int grid = team_grid(k_rkf45_tail, threads, smem, cap, cfg);
  k_rkf45_tail<<<grid, threads, smem, st>>>(d, p, y, dt, h_io, sp, steps, status, queue, list, count, cap);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ allocation-free ROS4
// Scratch of ck_integrate_ros4_noalloc: the work-queue counter that
// launch_ros4 otherwise receives from a per-call stream-ordered allocation.
// Every GPU that loads the library holds these 256 bytes until the process
// exits; all calls on a device share them.
static __device__ __align__(256) int32_t g_noalloc_scratch[NOALLOC_SCRATCH_INTS];

namespace {
std::mutex g_noalloc_mu;
int32_t* g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {};
}  // namespace

// Device address of g_noalloc_scratch on the current device.  The name is
// only a host-side stand-in, so the address is looked up once per device,
// with that device current, and cached.
cudaError_t noalloc_scratch(int32_t** out) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    g_noalloc_ptr[dev] = static_cast<int32_t*>(p);
  }
  *out = g_noalloc_ptr[dev];
  return cudaSuccess;
}

cudaError_t launch_ros4_noalloc(const HostMech& hm, int64_t n, const double* p, double* y,
                                const double* dt, double* h_io, const SolverParams& sp,
                                int32_t* steps, int32_t* status, cudaStream_t st,
                                const LaunchCfg& cfg) {
  if (cfg.precision) return cudaErrorNotSupported;  // its FP64 matrices need an allocation
  int32_t* queue = nullptr;
  cudaError_t e = noalloc_scratch(&queue);
  if (e != cudaSuccess) return e;
  // launch_ros4 zeroes the counter on the stream before the kernel starts;
  // no Jacobian copies (a rejected step recomputes J at the same state)
  return launch_ros4(hm, n, p, y, dt, h_io, sp, steps, status, queue, st, cfg, nullptr, 0, false);
}

}  // namespace ck
