// The ROS4 integrator kernel (Sec. 2 transformed form, App. C, driven by
// Algorithm 1): one CTA per reactor, iteration matrix in shared memory, and
// its launcher for one team size.  Included by one translation unit per team
// size (ck_ros4_*.cu).
#pragma once
#include <type_traits>

#include "ck_team_kernels.cuh"

namespace ck {

// Stage solve of the precision form: the iteration matrix is factored in
// FP32 (at the start of shared memory) and each solve is refined against the
// FP64 matrix M64 (the CTA's copy in global memory, L2-resident): x = LU32^-1
// b, then refine times r = b - M64 x (FP64), x += LU32^-1 r.  Arrays by offset
// in shared memory: b (in u) is overwritten with x; the second half of invd (n
// floats) and x (n doubles) are scratch.
static __device__ __noinline__ void refined_solve(const double* M64, int n, int rof_o, int invd_o, int u_o, int x_o,
                                                  int refine) {
  extern __shared__ __align__(16) double sm[];
  const int tid = threadIdx.x, P = blockDim.x, xf_o = 2 * invd_o + n;
  float* xf = reinterpret_cast<float*>(sm) + xf_o;
  double *u = sm + u_o, *x = sm + x_o;
  for (int i = tid; i < n; i += P) xf[i] = (float)u[i];
  team_sync();
  if (tid < 32) warp_solve<float>(0, n, rof_o, invd_o, xf_o);
  team_sync();
  for (int i = tid; i < n; i += P) x[i] = (double)xf[i];
  team_sync();
  for (int it = 0; it < refine; ++it) {
    // four lanes a row, one of four partial sums each (every fourth column;
    // the last n % 4 join the first), added as (s0 + s1) + (s2 + s3)
    const int n4 = n & ~3, q = tid & 3;
    for (int w = tid; w < ((4 * n + 31) & ~31); w += P) {
      const int i = w >> 2;
      double s = 0.0;
      if (i < n) {
        const double* row = M64 + (size_t)i * n;
        if (q == 0) s = u[i];
#pragma unroll 4
        for (int j = q; j < n4; j += 4) s = fma(-row[j], x[j], s);
        if (q == 0)
          for (int j = n4; j < n; ++j) s = fma(-row[j], x[j], s);
      }
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      s += __shfl_xor_sync(0xffffffffu, s, 2);
      if (q == 0 && i < n) xf[i] = (float)s;
    }
    team_sync();
    if (tid < 32) warp_solve<float>(0, n, rof_o, invd_o, xf_o);
    team_sync();
    for (int i = tid; i < n; i += P) x[i] += (double)xf[i];
    team_sync();
  }
  for (int i = tid; i < n; i += P) u[i] = x[i];
  team_sync();
}

// Step control, worked out by the first warp and read by all.
struct Ros4Ctl {
  double hh, dg;                          // step size, 1 / (hh gamma)
  double c21, c31, c32, c41, c42, c43;    // -c_ij / hh
  int go, accept;
};

// PREC 0: FP64 LU and solves.  PREC 1 / 2: FP32 LU and solves with one /
// two steps of FP64 iterative refinement (the rates, K_c, the temperature
// equation, the error norm and the step control stay FP64).
//
// P: threads of a team, at least n; the stage vectors are kept one component
// a thread, in registers.  MINB: resident teams an SM that the register
// allocation allows for.
//
// m64g (may be NULL for PREC 0) holds ros4_scratch_doubles(n) doubles per
// CTA, m64g[blockIdx.x][.]: global memory, 23 KB a CTA at n = 54 (21 MB for
// the 912 CTAs of the medium workload), so it stays in L2.  Its first n*n
// doubles hold J of the current state, its last n (precision form) the
// diagonal J_ii.
//
// The matrix factored is A = J - I/(h gamma) = -M rather than the iteration
// matrix M itself: partial pivoting picks the same rows, the multipliers and
// the pre-divided upper factor come out identical, and every solve returns
// exactly -u, so the stage vectors are kept as v_i = -u_i and the method's
// coefficients enter with their signs flipped.  The results are bitwise those
// of factoring M, without negating the n^2 entries of each new J.
//   - After a rejected step (error test, singular matrix or non-finite trial
//     state) y is unchanged, so J and f(y) are reused rather than recomputed
//     (only the analytic J: the forward-difference increments depend on h);
//     the new matrix J - I/(h gamma) is rebuilt from the copy.  With
//     m64g NULL (the allocation-free entry point) J is recomputed at the same
//     state instead, which gives the same values.
//   - The precision form keeps its FP64 iteration matrix, which the
//     refinement reads, in the first n*n doubles (the diagonal rebuilt from
//     the last n for each h) and its FP32 factors in the first half of the
//     shared FP64 matrix, so both forms need the same shared memory and
//     residency.
template <int P, int MINB, int PREC>
__global__ void __launch_bounds__(P, MINB) k_ros4(const __grid_constant__ DevMech d, int64_t N, const double* __restrict__ p,
                                                 double* __restrict__ y, const double* __restrict__ dt,
                                                 double* h_io, SolverParams sp, int32_t* steps,
                                                 int32_t* status, int32_t* queue, double* __restrict__ m64g) {
  extern __shared__ __align__(16) double sm[];
  __shared__ int slot;
  __shared__ Ros4Ctl ctl;
  constexpr bool INT = P == 256;               // products in integer arithmetic (see team_rhs)
  constexpr bool LAT = P == 128 && MINB == 4;  // right-hand sides in the latency form (team_rhs_lat)
  using F = typename std::conditional<PREC == 0, double, float>::type;  // type of the factors
  const int n = d.n, nn = n * n;
  const double* tab = d.tab;  // 2 KB, stays in L1
  const int ld = lu_ld(n);
  const float rc = 1.0f / (float)n;
  const Ros4Layout L(d, m64g != nullptr);
  double* M = sm;
  double* yv = sm + L.yv;
  double* F0 = sm + L.f0;
  double* Yt = sm + L.yt;
  double* ub = sm + L.ub;
  double* red = sm + L.bufs;
  F* MF = reinterpret_cast<F*>(M);         // PREC >= 1: FP32 factors over the FP64 matrix
  double* Mg = m64g ? m64g + (size_t)blockIdx.x * ros4_scratch_doubles(n) : nullptr;
  const bool keep_j = Mg != nullptr && sp.jac == 0;
  const bool fixed = sp.fixed_h > 0.0;
  const int tid = (int)threadIdx.x, warp = tid >> 5;
  const bool own = tid < n;
  for (;;) {
    const int r = team_next(queue, &slot);
    if (r >= N) break;
    if (own) yv[tid] = y[(int64_t)r * n + tid];
    const double pr = p[r];
    const double tf = dt[r];
    team_sync();
    int bad = own && !isfinite(yv[tid]);
    bad = __syncthreads_or(bad);
    bad |= !(pr > 0.0) || !isfinite(pr) || !(yv[0] > 0.0) || !isfinite(tf) || !(tf >= 0.0);
    // the first warp's view of the step control
    int st = ST_OK, acc = 0, rej = 0, sing_run = 0;
    double h = 0.0, t = 0.0, hh = 0.0;
    bool last_rej = false, last_nf = false, clamped = false;
    if (bad) {
      st = ST_BADINPUT;
    } else if (tf > 0.0) {
      if (fixed) h = sp.fixed_h;
      else if (h_io && h_io[r] > 0.0) h = h_io[r];
      else if (sp.h0 > 0.0) h = sp.h0;
      else h = team_h0<INT, LAT>(d, tab, pr, L.yv, tf, sp.rtol, sp.atol, L.f0, L.yt, L.ub, L.bufs, L.vp, L.rhs_q);
      const double hmin = 1e-15 * tf;
      // the next attempt: its step size, or the end of the integration
      auto next = [&](int accept) {
        int go = 0;
        if (t < tf) {
          if (acc + rej >= sp.max_steps) {
            st = ST_MAXSTEPS;
          } else {
            clamped = h >= tf - t;
            hh = clamped ? tf - t : h;
            if (hh < hmin) st = last_nf ? ST_NONFINITE : ST_HMIN;
            else go = 1;
          }
        }
        const double ih = rcp_rn(hh), dg = rcp_rn(hh * ROS_GAMMA);
        if (tid == 0) {
          ctl.hh = hh;
          ctl.dg = dg;
          ctl.c21 = -ROS_C21 * ih;
          ctl.c31 = -ROS_C31 * ih;
          ctl.c32 = -ROS_C32 * ih;
          ctl.c41 = -ROS_C41 * ih;
          ctl.c42 = -ROS_C42 * ih;
          ctl.c43 = -ROS_C43 * ih;
          ctl.go = go;
          ctl.accept = accept;
        }
      };
      if (warp == 0) next(0);
      bool have_j = false;   // J of yv in Mg (analytic form with a copy only)
      bool have_f = false;   // F0 = f(yv)
      team_sync();
      while (ctl.go) {
        // J and f at y (or the copy kept since a rejected attempt at the
        // same y); A = J - I/(hh gamma) = -M; LU of A
        if (!have_j) {
          if (sp.jac == 1) {
            team_jacobian_fd<INT, LAT>(d, tab, pr, L.yv, ctl.hh, sp.rtol, sp.atol, L.f0, PREC ? Mg : M, PREC ? n : ld, L.yt, L.ub, L.bufs, L.vp,
                             L.rhs_q, have_f);
          } else {
            // assembled in the copy Mg where there is one
            const JacTab& jt = Mg ? d.wide : d.narrow;
            team_jacobian<INT, LAT>(d, jt, tab, pr, yv, F0, Mg ? Mg : M, Mg && !PREC ? M : nullptr, ld,
                          carve_bufs(sm + L.bufs, d.S, sm + L.jscr, jt.chunk, L.vp));
          }
          if (PREC) {
            if (own) Mg[nn + tid] = Mg[(size_t)tid * n + tid];
            team_sync();
          }
          have_j = keep_j;
          have_f = true;
        } else if (PREC == 0) {
          for (int e = tid; e < nn; e += P) M[e + flat_row(e, rc) * (ld - n)] = Mg[e];
          team_sync();
        }
        if (PREC == 0) {
          if (own) M[tid * ld + tid] -= ctl.dg;
        } else {
          if (own) Mg[(size_t)tid * n + tid] = Mg[nn + tid] - ctl.dg;
          __syncthreads();
          for (int e = tid; e < nn; e += P) MF[e + flat_row(e, rc) * (ld - n)] = (F)Mg[e];
        }
        team_sync();
        const int info = team_lu<F>(0, n, L.rof, L.invd, L.lr, L.bufs + TEAM_RED_DOUBLES - 1);
        if (info) {
          if (warp == 0) {
            ++rej;
            if (++sing_run >= SINGULAR_LIMIT) {
              st = ST_SINGULAR;
              if (tid == 0) ctl.go = 0;
            } else {
              h = 0.5 * hh;
              last_rej = true;
              next(0);
            }
          }
          team_sync();
          continue;
        }
        auto solve = [&]() {  // ub <- A^-1 ub
          team_sync();
          if constexpr (PREC == 0) {
            if (warp == 0) warp_solve<double>(0, n, L.rof, L.invd, L.ub);
            team_sync();
          } else {
            refined_solve(Mg, n, L.rof, L.invd, L.ub, L.yt, PREC);
          }
        };
        double u1 = 0.0, u2 = 0.0, u3 = 0.0, u4 = 0.0, f3 = 0.0;
        const double yi = own ? yv[tid] : 0.0;
        // stage 1: M u1 = f(y), solved as A v1 = f(y) with v = -u (A = -M)
        if (own) ub[tid] = F0[tid];
        solve();
        // stage 2: M u2 = f(y + a21 u1) + (c21/h) u1
        if (own) {
          u1 = ub[tid];
          Yt[tid] = fma(-ROS_A21, u1, yi);
        }
        team_sync();
        team_rhs_any<INT, false, LAT>(d, tab, pr, L.yt, L.ub, L.bufs, L.vp, L.rhs_q);
        if (own) ub[tid] = fma(ctl.c21, u1, ub[tid]);
        solve();
        // stage 3: M u3 = f(y + a31 u1 + a32 u2) + (c31 u1 + c32 u2)/h
        if (own) {
          u2 = ub[tid];
          Yt[tid] = fma(-ROS_A32, u2, fma(-ROS_A31, u1, yi));
        }
        team_sync();
        team_rhs_any<INT, false, LAT>(d, tab, pr, L.yt, L.ub, L.bufs, L.vp, L.rhs_q);
        if (own) {
          f3 = ub[tid];
          ub[tid] = fma(ctl.c32, u2, fma(ctl.c31, u1, f3));
        }
        solve();
        // stage 4: same argument as stage 3 (a4j = a3j, a43 = 0), so f is reused
        if (own) {
          u3 = ub[tid];
          ub[tid] = fma(ctl.c43, u3, fma(ctl.c42, u2, fma(ctl.c41, u1, f3)));
        }
        solve();
        // y* = y + sum m_i u_i, e = sum E_i u_i; u_i = -v_i; the norm
        // sqrt(mean (e_i / (atol + rtol max(|y_i|, |y*_i|)))^2)
        double yn = 0.0, s = 0.0;
        if (own) {
          u4 = ub[tid];
          yn = fma(-ROS_M4, u4, fma(-ROS_M3, u3, fma(-ROS_M2, u2, fma(-ROS_M1, u1, yi))));
          const double e = fma(-ROS_E4, u4, fma(-ROS_E3, u3, fma(-ROS_E2, u2, -ROS_E1 * u1)));
          if (!fixed) {
            const double v = e / (sp.atol + sp.rtol * fmax(fabs(yi), fabs(yn)));
            s = __dmul_rn(v, v);
          }
        }
        if (32 * warp < n) {
          s = warp_allsum(s);
          if ((tid & 31) == 0) red[warp] = s;
        }
        const int nf = __syncthreads_or(own && !isfinite(yn));
        if (warp == 0) {
          int accept = 1;
          if (fixed) {
            t = clamped ? tf : t + hh;
            ++acc;
          } else {
            double q = 0.0;
            for (int g = 0; 32 * g < n; ++g) q += red[g];
            const double e = sqrt(q / n);
            if (nf || !isfinite(e)) {
              ++rej;
              h = FAC_MIN * hh;
              last_rej = true;
              last_nf = true;
              accept = 0;
            } else {
              last_nf = false;
              const double pe = (e == 0.0) ? 0.0 : pow(e, -0.25);
              if (e < 1.0) {
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
                accept = 0;
              }
            }
          }
          sing_run = 0;
          next(accept);
        }
        team_sync();
        if (ctl.accept) {
          if (own) yv[tid] = yn;
          have_j = have_f = false;
        }
        team_sync();
      }
    }
    team_sync();
    if (own) y[(int64_t)r * n + tid] = yv[tid];
    if (tid == 0) {
      if (h_io && st != ST_BADINPUT && tf > 0.0) h_io[r] = h;
      if (steps) {
        steps[2 * (int64_t)r] = acc;
        steps[2 * (int64_t)r + 1] = rej;
      }
      status[r] = st;
    }
    team_sync();
  }
}

// Launch k_ros4<P, MINB, precision> (the body of launch_ros4 for one team
// size; each is compiled in its own translation unit).
template <int P, int MINB>
cudaError_t launch_ros4_team(const HostMech& hm, int64_t n, const double* p, double* y, const double* dt,
                             double* h_io, const SolverParams& sp, int32_t* steps, int32_t* status,
                             int32_t* queue, cudaStream_t st, const LaunchCfg& cfg, double* scratch,
                             size_t scratch_bytes, bool may_alloc) {
  const int nn = hm.d.n;
  auto kern = cfg.precision == 2 ? k_ros4<P, MINB, 2>
                                 : (cfg.precision == 1 ? k_ros4<P, MINB, 1> : k_ros4<P, MINB, 0>);
  // with at most one reactor an SM, all rates of progress at once
  DevMech d = hm.d;
  if (n <= sm_count() && hm.R > 0) {
    d.rhs_chunk = hm.R;
    if (Ros4Layout(d, true).doubles > (size_t)smem_doubles(1)) d.rhs_chunk = hm.d.rhs_chunk;
  }
  size_t smem = sizeof(double) * Ros4Layout(d, true).doubles;
  int grid = team_grid(kern, P, smem, n, cfg);
  // per-CTA copies of J (every form) and the FP64 iteration matrices of
  // the precision form: the caller's scratch when it is large enough, else
  // a stream-ordered allocation around the launch, else (allocation-free
  // FP64 form) none
  const size_t need = sizeof(double) * (size_t)grid * ros4_scratch_doubles(nn);
  double* m64g = nullptr;
  bool owned = false;
  if (scratch && scratch_bytes >= need) {
    m64g = scratch;
  } else if (may_alloc) {
    cudaError_t a = cudaMallocAsync(reinterpret_cast<void**>(&m64g), need, st);
    if (a != cudaSuccess) return a;
    owned = true;
  } else if (cfg.precision) {
    return cudaErrorNotSupported;
  } else {
    smem = sizeof(double) * Ros4Layout(d, false).doubles;
    grid = team_grid(kern, P, smem, n, cfg);
  }
  kern<<<grid, P, smem, st>>>(d, n, p, y, dt, h_io, sp, steps, status, queue, m64g);
  cudaError_t k = cudaGetLastError();
  if (owned) {
    cudaError_t f = cudaFreeAsync(m64g, st);
    if (k == cudaSuccess) k = f;
  }
  return k;
}

}  // namespace ck
