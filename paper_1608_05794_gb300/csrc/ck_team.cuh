// Team-per-reactor device code: one CTA (1..8 warps) evaluates one reactor's
// right-hand side and analytic Jacobian, and factors and solves its
// iteration matrix I/(h gamma) - J held in shared memory (Sec. 2, ROS4).
// This is the paper's "deep" vectorisation (Sec. 4): lanes split the
// reactions and species of a single ODE system.  All sums that feed a
// control decision are reduced in a fixed order, so every thread of the CTA
// takes the same branch and results are bitwise reproducible.
#pragma once
#include "ck_common.cuh"
#include "ck_layout.cuh"

namespace ck {

__device__ __forceinline__ double warp_allsum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block-wide sum returned to every thread (fixed order).  red: >= 32 doubles.
__device__ __forceinline__ double team_sum(double v, double* red) {
  v = warp_allsum(v);
  const int nw = blockDim.x >> 5;
  if (nw == 1) return v;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  for (int i = 0; i < nw; ++i) s += red[i];
  return s;
}

// Butterfly sums of 2, 4 or 8 values over the 32 lanes of a warp, packed:
// after the first exchange each half of the warp carries half of the values,
// and so on, so that 4 sums cost 6 adds instead of 20 (an FP64 add costs the
// warp 64 cycles of its pipe however few lanes carry something useful).
// Every value is summed by the same tree as warp_allsum (strides 16, 8, 4,
// 2, 1; only the order of the two operands of an add may differ), so the sums
// are bitwise those of warp_allsum.  The sum of value q ends in every lane
// whose leading lane bits (16 first) spell q: lane q * (32 / N) holds it.
__device__ __forceinline__ double pack_step(double keep_lo, double keep_hi, int o) {
  const bool hi = (threadIdx.x & o) != 0;
  return (hi ? keep_hi : keep_lo) + __shfl_xor_sync(0xffffffffu, hi ? keep_lo : keep_hi, o);
}
__device__ __forceinline__ double warp_sum_pack2(double a, double b) {
  double v = pack_step(a, b, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_sum_pack4(double a, double b, double c, double d) {
  double v = pack_step(pack_step(a, c, 16), pack_step(b, d, 16), 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_sum_pack8(const double (&a)[8]) {
  const double p0 = pack_step(a[0], a[4], 16), p1 = pack_step(a[1], a[5], 16);
  const double p2 = pack_step(a[2], a[6], 16), p3 = pack_step(a[3], a[7], 16);
  double v = pack_step(pack_step(p0, p2, 8), pack_step(p1, p3, 8), 4);
#pragma unroll
  for (int o = 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// A sum over the species taken by one warp: g[q] holds the part of lanes 32 q
// to 32 q + 31 of a team of b.vp threads; the parts are summed each by the
// warp tree and then in order, as team_sum does.  ng parts (1..4), the rest
// must be zero.  The total reaches every lane.
__device__ __forceinline__ double warp_sum_groups(const double (&g)[4], int ng) {
  if (ng == 1) return warp_allsum(g[0]);
  if (ng == 2) {
    const double v = warp_sum_pack2(g[0], g[1]);
    return __shfl_sync(0xffffffffu, v, 0) + __shfl_sync(0xffffffffu, v, 16);
  }
  const double v = warp_sum_pack4(g[0], g[1], g[2], g[3]);
  double s = __shfl_sync(0xffffffffu, v, 0) + __shfl_sync(0xffffffffu, v, 8);
  s += __shfl_sync(0xffffffffu, v, 16);
  if (ng > 3) s += __shfl_sync(0xffffffffu, v, 24);
  return s;
}

__device__ __forceinline__ void team_sync() {
  if (blockDim.x == 32) __syncwarp();
  else __syncthreads();
}

// Shared-memory work arrays of one team (species_doubles: [red | X Gp Gm hRT |
// cpR | wd]; a Jacobian continues with aT E u).
// The Jacobian processes reactions in the chunks of its table (JacTab); the
// right-hand side, which keeps one value per reaction, takes all reactions at
// once or chunks of m.rhs_chunk.  Gp_k = 2^(g_k) and Gm_k = 2^(-g_k) with g_k =
// (S/R - H/RT)_k / ln 2, so that 1/K_c of Eq. kc is a product of species
// factors.  Entry S of X, Gp, Gm (1) and hRT (0) stands for an empty reaction
// slot.  After the reaction passes of the Jacobian, X, Gp and Gm are reused
// (dense, cs, eW).
struct TeamBufs {
  double *X, *Gp, *Gm, *hRT;              // [S + 1]
  double *cpR, *wd, *aT, *E, *u;          // [S]; wd, aT, E, u contiguous
  double *q, *dqT, *D, *P, *w;            // per-reaction values of a chunk (JAC_PER_RXN)
  double* red;                            // [TEAM_RED_DOUBLES] reductions and scalars (SC_*)
  int vp;                                 // lanes that the species sums are grouped by (64 or 256)
};

__device__ __forceinline__ TeamBufs carve_bufs(double* base, int S, double* scratch, int chunk, int vp) {
  TeamBufs b;
  b.red = base;
  b.X = b.red + TEAM_RED_DOUBLES;
  b.Gp = b.X + S + 1;
  b.Gm = b.Gp + S + 1;
  b.hRT = b.Gm + S + 1;
  b.cpR = b.hRT + S + 1;
  b.wd = b.cpR + S;
  b.aT = b.wd + S;
  b.E = b.aT + S;
  b.u = b.E + S;
  b.q = scratch;
  b.dqT = b.q + chunk;
  b.D = b.dqT + chunk;
  b.P = b.D + chunk;
  b.w = b.P + 6 * chunk;
  b.vp = vp;
  return b;
}

// Scalars of one evaluation, formed once by one warp (an FP64 instruction
// costs every warp that issues it a full slot) and read by all from red[].
enum : int {
  SC_INVT = 32, SC_LNT, SC_LOG2T, SC_T2, SC_T3, SC_T4,  // functions of T
  SC_PW,                                                // (R T / p0)^dnu, dnu = -2..2
  SC_WBAR = SC_PW + 5, SC_RHO, SC_INVRHO, SC_CTOT,      // mixture
  SC_TDOT, SC_ICPM, SC_POW,
  SC_SUM = 52                                           // the Jacobian's seven species sums
};

// Mixture quantities shared by the RHS and the Jacobian.
struct Mix {
  double T, invT, log2T, rho, invrho, Wbar, Ctot;
};

// Groups of 32 species (at most 4).
__device__ __forceinline__ int species_groups(int S) { return (S + 31) >> 5; }

// Species pass: rho, [X_k], Gibbs / enthalpy / heat-capacity polynomials.
// The mixture (a chain of sums and divisions) and the functions of T (a chain
// through log T) are formed side by side by two warps, everything else of
// the species by all of them: a polynomial pass of 32 species is one work
// item, dealt to the warps in turn.
// Ends with a barrier and returns (the same in every thread) whether the
// ranges allow the reactions' products to be taken in integer arithmetic
// (mul_int).
// ORD: the species sums one species after another, as the threads of RKF45 take
// them (rhs_thread without TEAM), instead of by trees.
template <bool ORD, bool INT>
__device__ __forceinline__ bool team_species(const DevMech& m, double p, const double* y,
                                             TeamBufs& b, Mix& x, const double* tab) {
  const int S = m.S, tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const int SG = species_groups(S);
  double* red = b.red;
  const double T = y[0];
  x.T = T;
  bool ok = temp_in_range(T);
  if (warp == nw - 1) {
    const double invT = rcp_sel<INT>(T), lnT = log(T);
    const double T2 = T * T, T3 = T2 * T;
    const double up = T * R_OVER_P0, dn = invT * P0_OVER_R;
    if (lane == 0) {
      red[SC_INVT] = invT;
      red[SC_LNT] = lnT;
      red[SC_LOG2T] = lnT * INV_LN2;
      red[SC_T2] = T2;
      red[SC_T3] = T3;
      red[SC_T4] = T3 * T;
      red[SC_PW] = dn * dn;
      red[SC_PW + 1] = dn;
      red[SC_PW + 2] = 1.0;
      red[SC_PW + 3] = up;
      red[SC_PW + 4] = up * up;
    }
  }
  if (warp == 0) {
    double yw[4], part[4] = {0.0, 0.0, 0.0, 0.0};
    const bool fold = b.vp == 64;  // species 64 + t joins species t in its lane's part
    const int ng = fold && SG > 2 ? 2 : SG;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      yw[q] = 0.0;
      if (q < SG) {
        const int k = 32 * q + lane;
        const double yk = k < S ? y[1 + k] : 0.0, iw = k < S ? m.invW[k] : 0.0;
        yw[q] = __dmul_rn(yk, iw);  // (rounded: a sum over lanes must not take the product in)
        if (q >= 2 && fold) part[q - 2] = fma(yk, iw, part[q - 2]);
        else part[q] = yw[q];
      }
    }
    double sumYW = 0.0;
    if (ORD) {
      for (int k = 0; k < S; ++k) sumYW = fma(y[1 + k], m.invW[k], sumYW);
    } else {
      sumYW = warp_sum_groups(part, ng);
    }
    const double Wbar = rcp_sel<INT>(sumYW);
    const double rho = m.cv ? p : p / (R_GAS * T * sumYW);  // constant volume: p is the density
    const double invrho = rcp_sel<INT>(rho);
#pragma unroll
    for (int q = 0; q < 4; ++q) part[q] = 0.0;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q < SG) {
        const int k = 32 * q + lane;
        const double xk = k < S ? __dmul_rn(rho, yw[q]) : 0.0;
        if (k < S) {
          b.X[k] = xk;
          ok &= conc_in_range(xk);
        }
        if (q >= 2 && fold) part[q - 2] += xk;
        else part[q] = xk;
      }
    double Ctot = 0.0;
    if (ORD) {
      __syncwarp();
      for (int k = 0; k < S; ++k) Ctot += b.X[k];
    } else {
      Ctot = warp_sum_groups(part, ng);
    }
    if (lane == 0) {
      red[SC_WBAR] = Wbar;
      red[SC_RHO] = rho;
      red[SC_INVRHO] = invrho;
      red[SC_CTOT] = Ctot;
      b.X[S] = b.Gp[S] = b.Gm[S] = 1.0;
      b.hRT[S] = 0.0;
    }
  }
  team_sync();
  x.invT = red[SC_INVT];
  x.log2T = red[SC_LOG2T];
  x.Wbar = red[SC_WBAR];
  x.rho = red[SC_RHO];
  x.invrho = red[SC_INVRHO];
  x.Ctot = red[SC_CTOT];
  const double lnT = red[SC_LNT], T2 = red[SC_T2], T3 = red[SC_T3], T4 = red[SC_T4];
  for (int it = warp; it < 2 * SG; it += nw) {
    const bool gibbs = it < SG;
    const int k = 32 * (gibbs ? it : it - SG) + lane;
    if (k < S) {
      const double* a = m.thermo + k * TH_PER_SPECIES + (T < m.tmid[k] ? 0 : TH_STRIDE);
      if (gibbs) {
        double g = fma(a[11], lnT, a[12]);
        g = fma(a[13], T, g);
        g = fma(a[14], T2, g);
        g = fma(a[15], T3, g);
        g = fma(a[16], T4, g);
        g = fma(a[17], x.invT, g);
        ok &= gibbs_in_range(g);
        ck_exp2_pm(g, tab, b.Gp[k], b.Gm[k]);
      } else {
        b.cpR[k] = fma(a[4], T4, fma(a[3], T3, fma(a[2], T2, fma(a[1], T, a[0]))));
        b.hRT[k] = fma(a[10], x.invT, fma(a[9], T4, fma(a[8], T3, fma(a[7], T2, fma(a[6], T, a[5])))));
      }
    }
  }
  return __syncthreads_and(ok);
}

// A reaction record without its fall-off limit (the last two vectors) in
// 16-byte loads; the fields are then read from registers.
__device__ __forceinline__ RxnRec load_rxn(const RxnRec* src) {
  RxnRec r;
  const int4* s = reinterpret_cast<const int4*>(src);
  int4* t = reinterpret_cast<int4*>(&r);
#pragma unroll
  for (int q = 0; q < 5; ++q) t[q] = __ldg(s + q);
  return r;
}

// Rates of one reaction at the mixture state.  JAC: also the partial-
// derivative pieces used by the Jacobian (see team_jacobian).  i: index of
// the reaction inside the current chunk, iw: among its typed reactions.
// Empty slots read the neutral entries of the species arrays (a product with
// 1, a sum with 0, exact), so that reactions of every molecularity take the
// same instructions.  INT: the products of concentrations and of Gibbs factors
// in integer arithmetic, beside the FP64 unit, which bounds the team kernels
// (10 of the 23 FP64 instructions of a rate, 20 of 49 with its derivatives).
// ORD: the fall-off factor by a division, as RKF45's threads form it.  PRE: k_f
// is at hand in b.q[i], and in b.w[iw] k_0/k_inf (JAC) or the whole factor of the
// net rate (team_species_lat).
template <bool JAC, bool INT, bool ORD = false, bool PRE = false>
__device__ __forceinline__ void team_reaction(const DevMech& m, const RxnRec* src, const Mix& x,
                                              const TeamBufs& b, const double* tab, int i, int iw) {
  const RxnRec r = load_rxn(src);
  const double* X = b.X;
  const double l2kf = fma(-r.EoR2, x.invT, fma(r.beta, x.log2T, r.lA2));
  const double kf = PRE ? b.q[i] : ck_exp2(l2kf, tab);
  const int s0 = r.sp[0], s1 = r.sp[1], s2 = r.sp[2], s3 = r.sp[3], s4 = r.sp[4], s5 = r.sp[5];
  const double x0 = X[s0], x1 = X[s1], x2 = X[s2], y0 = X[s3], y1 = X[s4], y2 = X[s5];
  const double fwd = mul_sel<INT>(mul_sel<INT>(x0, x1), x2);
  double kr = 0.0, rv = 0.0, dlnkc = 0.0;
  if (r.rev == 2) {
    // explicit reverse Arrhenius; for the Jacobian, d ln k_r/dT enters as
    // d ln k_f/dT - d ln K_c/dT, so dlnkc carries their difference
    const double* ra = m.revp + 3 * r.rev_ix;
    kr = ck_exp2(fma(-ra[2], x.invT, fma(ra[1], x.log2T, ra[0])), tab);
    rv = mul_sel<INT>(mul_sel<INT>(y0, y1), y2);
    if (JAC) {
      const double dlnkf = fma(r.EoR, x.invT, r.beta) * x.invT;
      dlnkc = dlnkf - fma(ra[2] * LN2, x.invT, ra[1]) * x.invT;
    }
  } else if (r.rev) {
    // 1/K_c = (R T/p0)^dnu prod_reactants Gp prod_products Gm (Eq. kc)
    double kci = mul_sel<INT>(b.red[SC_PW + 2 + r.dnu], b.Gp[s0]);
    kci = mul_sel<INT>(kci, b.Gm[s3]);
    kci = mul_sel<INT>(kci, b.Gp[s1]);
    kci = mul_sel<INT>(kci, b.Gm[s4]);
    kci = mul_sel<INT>(kci, b.Gp[s2]);
    kci = mul_sel<INT>(kci, b.Gm[s5]);
    kr = kf * kci;
    rv = mul_sel<INT>(mul_sel<INT>(y0, y1), y2);
    if (JAC) {
      // d ln K_c / dT = (sum_j nu_j H_j/(R T) - dnu) / T
      double hs = b.hRT[s3];
      hs += b.hRT[s4];
      hs += b.hRT[s5];
      hs -= b.hRT[s0];
      hs -= b.hRT[s1];
      hs -= b.hRT[s2];
      dlnkc = (hs - r.dnu_d) * x.invT;
    }
  }
  const double net = fma(-kr, rv, kf * fwd);
  double q = net, ckf = kf, ckr = kr, w = 0.0, M = 0.0, dcdT = 0.0;
  const double dlnkf = fma(r.EoR, x.invT, r.beta) * x.invT;
  if (PRE && !JAC) {
    b.q[i] = r.type ? b.w[iw] * net : net;
    return;
  }
  if (r.type) {
    double c, dcdM;
    M = x.Ctot;
    for (int e = r.eff_beg; e < r.eff_beg + r.eff_cnt; ++e) M = fma(m.eff_m1[e], X[m.eff_sp[e]], M);
    if (r.type == 1) {
      c = M;
      dcdM = 1.0;
    } else {
      const double2 f0 = __ldg(reinterpret_cast<const double2*>(src) + 5);  // lA02, beta0
      const double2 f1 = __ldg(reinterpret_cast<const double2*>(src) + 6);  // E0oR2, E0oR
      const double l2k0 = fma(-f1.x, x.invT, fma(f0.y, x.log2T, f0.x));
      const double k0_kf = PRE ? b.w[iw] : ck_exp2(l2k0 - l2kf, tab);
      const double Pr = __dmul_rn(k0_kf, M);
      if (ORD) {
        b.q[i] = net * (Pr / (1.0 + Pr));
        return;
      }
      const double inv1p = rcp_rn(__dadd_rn(1.0, Pr));
      c = Pr * inv1p;
      dcdM = k0_kf * inv1p * inv1p;
      if (JAC) {
        const double dlnk0 = fma(f1.y, x.invT, f0.y) * x.invT;
        const double ds = fma(fma(f1.y, x.invT, f0.y), x.invT, -dlnkf);
        dcdT = Pr * ds * inv1p * inv1p;
      }
    }
    q = c * net;
    if (JAC) {
      ckf = c * kf;
      ckr = c * kr;
      w = dcdM * net;
      b.w[iw] = w;
    }
  }
  b.q[i] = q;
  if (JAC) {
    // d q / d[X] slot by slot: c k_f prod of the other reactant slots, and
    // -c k_r prod of the other product slots
    double* P = b.P + 6 * i;
    const double x12 = mul_sel<INT>(x1, x2), x02 = mul_sel<INT>(x0, x2), x01 = mul_sel<INT>(x0, x1);
    const double y12 = mul_sel<INT>(y1, y2), y02 = mul_sel<INT>(y0, y2), y01 = mul_sel<INT>(y0, y1);
    const bool in = INT && rate_in_range(ckf) && (!r.rev || rate_in_range(ckr));
    if (INT && __all_sync(__activemask(), in)) {
      P[0] = mul_sel<INT>(ckf, x12);
      P[1] = mul_sel<INT>(ckf, x02);
      P[2] = mul_sel<INT>(ckf, x01);
      if (r.rev) {
        P[3] = mul_sel<INT>(-ckr, y12);
        P[4] = mul_sel<INT>(-ckr, y02);
        P[5] = mul_sel<INT>(-ckr, y01);
      }
    } else {
      P[0] = ckf * x12;
      P[1] = ckf * x02;
      P[2] = ckf * x01;
      if (r.rev) {
        P[3] = -ckr * y12;
        P[4] = -ckr * y02;
        P[5] = -ckr * y01;
      }
    }
    // D = sum_j dq/d[X_j] [X_j]: Euler's theorem for the mass-action
    // products (homogeneous of degree nreac / nprod) plus the [M] part.
    double D = fma(ckf * fwd, r.nreac_d, -(ckr * rv) * r.nprod_d);
    // dq/dT at fixed [X], then the total derivative at fixed Y (d[X]/dT =
    // -[X]/T at constant pressure, 0 at constant volume)
    const double tA = __dmul_rn(ckf, fwd), tB = __dmul_rn(ckr, rv);
    double dqTX = fma(tA, dlnkf, -__dmul_rn(tB, __dadd_rn(dlnkf, -dlnkc)));
    if (r.type) {
      D = fma(M, w, D);
      dqTX = fma(dcdT, net, dqTX);
    }
    b.D[i] = D;
    b.dqT[i] = m.cv ? dqTX : fma(-D, x.invT, dqTX);
  }
}

// Named barriers of the first 128 threads' teams: `sync` waits until n threads
// have come, `arrive` counts the caller's warp without waiting.
__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int n) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// team_species for a team of four warps on a mechanism of at most 32 species,
// arranged for the shortest chain: one warp issues an FP64 instruction every
// 68 cycles however independent they are, so that every warp takes its own
// share: warp 1 log T, warp 2 1/T and the powers; then, without waiting for
// the mixture, warp 3 the Gibbs factors, warp 1 the heat capacities and
// enthalpies, warp 2 the rate constants k_f (kf[R]), which need T alone; warp 0
// the mixture and, of the third-body and fall-off reactions, k_0/k_inf (k0,
// JAC) or the whole factor that multiplies their net rate (k0, else).  JAC: the
// mean molar mass too.  The same values as team_species and team_reaction.
template <bool ORD, bool JAC>
__device__ __forceinline__ void team_species_lat(const DevMech& m, double p, const double* y, TeamBufs& b, Mix& x,
                                                 const double* tab, double* kf, double* k0) {
  const int S = m.S, R = m.R, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double* red = b.red;
  const double T = y[0];
  const bool in = lane < S;
  x.T = T;
  if (warp == 0) {
    const double yw = in ? __dmul_rn(y[1 + lane], m.invW[lane]) : 0.0;
    double sumYW = 0.0;
    if (ORD) {
      for (int k = 0; k < S; ++k) sumYW = fma(y[1 + k], m.invW[k], sumYW);
    } else {
      sumYW = warp_allsum(yw);
    }
    const double rho = m.cv ? p : p / (R_GAS * T * sumYW);
    const double xk = in ? __dmul_rn(rho, yw) : 0.0;
    if (in) b.X[lane] = xk;
    if (lane == 0) {
      red[SC_RHO] = rho;
      b.X[S] = b.Gp[S] = b.Gm[S] = 1.0;
      b.hRT[S] = 0.0;
    }
    __syncwarp();
    double c = 0.0;
    if (ORD) {
      for (int k = 0; k < S; ++k) c += b.X[k];
    } else {
      c = warp_allsum(xk);
    }
    if (lane == 0) red[SC_CTOT] = c;
    if (JAC) {
      const double Wbar = rcp_rn(sumYW), invrho = rcp_rn(rho);
      if (lane == 0) {
        red[SC_WBAR] = Wbar;
        red[SC_INVRHO] = invrho;
      }
    }
    bar_sync(2, 96);  // the functions of T, from warps 1 and 2
    for (int i = m.first_typed + lane; i < R; i += 32) {
      const RxnRec* src = m.rxn + i;
      const bool fall = src->type == 2;
      double k0kf = 0.0;
      if (fall) {
        const double l2kf = fma(-src->EoR2, red[SC_INVT], fma(src->beta, red[SC_LOG2T], src->lA2));
        const double l2k0 = fma(-src->E0oR2, red[SC_INVT], fma(src->beta0, red[SC_LOG2T], src->lA02));
        k0kf = ck_exp2(l2k0 - l2kf, tab);
      }
      if (!JAC) {
        double M = c;
        for (int e = src->eff_beg; e < src->eff_beg + src->eff_cnt; ++e) M = fma(m.eff_m1[e], b.X[m.eff_sp[e]], M);
        if (fall) {
          const double Pr = __dmul_rn(k0kf, M);
          k0kf = ORD ? Pr / __dadd_rn(1.0, Pr) : __dmul_rn(Pr, rcp_rn(__dadd_rn(1.0, Pr)));
        } else {
          k0kf = M;
        }
      }
      k0[i - m.first_typed] = k0kf;
    }
  } else {
    if (warp == 1) {
      const double lnT = log(T);
      if (lane == 0) {
        red[SC_LNT] = lnT;
        red[SC_LOG2T] = lnT * INV_LN2;
      }
      bar_arrive(2, 96);
    } else if (warp == 2) {
      const double invT = rcp_rn(T), T2 = T * T, T3 = T2 * T;
      const double up = T * R_OVER_P0, dn = invT * P0_OVER_R;
      if (lane == 0) {
        red[SC_INVT] = invT;
        red[SC_T2] = T2;
        red[SC_T3] = T3;
        red[SC_T4] = T3 * T;
        red[SC_PW] = dn * dn;
        red[SC_PW + 1] = dn;
        red[SC_PW + 2] = 1.0;
        red[SC_PW + 3] = up;
        red[SC_PW + 4] = up * up;
      }
      bar_arrive(2, 96);
    }
    bar_sync(1, 96);  // warps 1 to 3
    const double invT = red[SC_INVT], log2T = red[SC_LOG2T];
    const double T2 = red[SC_T2], T3 = red[SC_T3], T4 = red[SC_T4];
    const double* a = m.thermo + lane * TH_PER_SPECIES + (in && T < m.tmid[lane] ? 0 : TH_STRIDE);
    if (warp == 3 && in) {
      double g = fma(a[11], red[SC_LNT], a[12]);
      g = fma(a[13], T, g);
      g = fma(a[14], T2, g);
      g = fma(a[15], T3, g);
      g = fma(a[16], T4, g);
      g = fma(a[17], invT, g);
      ck_exp2_pm(g, tab, b.Gp[lane], b.Gm[lane]);
    } else if (warp == 1 && in) {
      b.cpR[lane] = fma(a[4], T4, fma(a[3], T3, fma(a[2], T2, fma(a[1], T, a[0]))));
      b.hRT[lane] = fma(a[10], invT, fma(a[9], T4, fma(a[8], T3, fma(a[7], T2, fma(a[6], T, a[5])))));
    } else if (warp == 2) {
      for (int i = lane; i < R; i += 32) {
        const RxnRec* src = m.rxn + i;
        kf[i] = ck_exp2(fma(-src->EoR2, invT, fma(src->beta, log2T, src->lA2)), tab);
      }
    }
  }
  __syncthreads();
  x.invT = red[SC_INVT];
  x.log2T = red[SC_LOG2T];
  x.rho = red[SC_RHO];
  x.Ctot = red[SC_CTOT];
  x.Wbar = JAC ? red[SC_WBAR] : 0.0;
  x.invrho = JAC ? red[SC_INVRHO] : 0.0;
}

// The reaction that place s of a team's walk over R reactions takes, or -1:
// elementary reactions first, the others from a warp of their own on, so that
// the two kinds run side by side.
__device__ __forceinline__ int lat_slots(int R, int ft) { return ((ft + 31) & ~31) + R - ft; }
__device__ __forceinline__ int lat_reaction(int s, int ft) {
  const int es = (ft + 31) & ~31;
  return s < ft ? s : (s >= es ? ft + s - es : -1);
}

// team_rhs arranged like team_species_lat (four warps, at most 32 species, q of
// m.R doubles and one more for each third-body or fall-off reaction).  ORD: see
// team_rhs.  The same values.  RKF45 on 2000 reactors of the 10-species
// mechanism, whose time is that of the longest: 42.6 ms, with team_rhs on two
// warps 50.8.
template <bool ORD>
static __device__ __noinline__ void team_rhs_lat(const DevMech& m, const double* tab, double p, int y_o, int f_o,
                                                 int bufs_o, int q_o) {
  extern __shared__ __align__(16) double sm[];
  const double* y = sm + y_o;
  double* f = sm + f_o;
  TeamBufs b = carve_bufs(sm + bufs_o, m.S, sm + q_o, 0, 64);
  b.w = b.q + m.R;
  Mix x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, S = m.S;
  team_species_lat<ORD, false>(m, p, y, b, x, tab, b.q, b.w);
  for (int s = threadIdx.x; s < lat_slots(m.R, m.first_typed); s += blockDim.x) {
    const int i = lat_reaction(s, m.first_typed);
    if (i >= 0) team_reaction<false, false, ORD, true>(m, m.rxn + i, x, b, tab, i, i - m.first_typed);
  }
  if (warp == 3) {  // rho c_p meanwhile
    double c = 0.0, yk = 0.0;
    if (lane < S) {
      c = m.cv ? b.cpR[lane] - 1.0 : b.cpR[lane];
      yk = __dmul_rn(y[1 + lane], m.invW[lane]);
    }
    double cpm = 0.0;
    if (ORD) {
      for (int k = 0; k < S; ++k) cpm = fma(__shfl_sync(0xffffffffu, yk, k), __shfl_sync(0xffffffffu, c, k), cpm);
    } else {
      cpm = warp_allsum(fma(yk, c, 0.0));
    }
    if (lane == 0) b.red[SC_ICPM] = x.rho * cpm;
  } else if (warp == 2) {  // and 1 / rho
    const double invrho = rcp_rn(x.rho);
    if (lane == 0) b.red[SC_INVRHO] = invrho;
  }
  // the gather's terms are read ahead of the rates
  constexpr int PF = 8;
  const int32_t* ptr = ORD ? m.slot_ptr : m.csr_ptr;
  const CsrTerm* terms = ORD ? m.slot : m.csr;
  int e = 0, e1 = 0;
  CsrTerm t[PF];
  if (warp == 0 && lane < S) {
    e = ptr[lane];
    e1 = ptr[lane + 1];
#pragma unroll
    for (int u = 0; u < PF; ++u)
      if (e + u < e1) t[u] = terms[e + u];
  }
  __syncthreads();
  if (warp == 0) {
    double w = 0.0, h = 0.0;
    if (lane < S) {
      while (e < e1) {
        double q[PF];
#pragma unroll
        for (int u = 0; u < PF; ++u) q[u] = e + u < e1 ? b.q[t[u].rx] : 0.0;
#pragma unroll
        for (int u = 0; u < PF; ++u)
          if (e + u < e1) w = fma(t[u].nu, q[u], w);
        e += PF;
#pragma unroll
        for (int u = 0; u < PF; ++u)
          if (e + u < e1) t[u] = terms[e + u];
      }
      f[1 + lane] = w * (m.W[lane] * b.red[SC_INVRHO]);
      h = m.cv ? b.hRT[lane] - 1.0 : b.hRT[lane];
    }
    double hw = 0.0;
    if (ORD) {
      for (int k = 0; k < S; ++k) hw = fma(__shfl_sync(0xffffffffu, h, k), __shfl_sync(0xffffffffu, w, k), hw);
    } else {
      hw = warp_allsum(fma(h, w, 0.0));
    }
    if (lane == 0) f[0] = -x.T * hw / b.red[SC_ICPM];
  }
  __syncthreads();
}

// f(y) for one reactor.  Arrays by their offsets (doubles) in the CTA's
// dynamic shared memory, so that this out-of-line function still addresses
// shared memory directly: y_o, f_o the vectors (n = S + 1; f may not be y),
// bufs_o the work arrays (species_doubles), qq the rates of progress.
// INT: products in integer arithmetic where the ranges allow it.  That pays
// where the FP64 unit is the bound (RKF45 on 16384 reactors of the 53-species
// mechanism: 278 against 321 ms), not where a team waits for its chain of
// operations (a product is 106 cycles of it in integers, 72 in FP64: ROS4 on
// 512 reactors of the 10-species mechanism, 245 against 230 ms) or is short of
// registers (ROS4 on 4096 of the 53-species one, 617 against 600 ms).
// ORD: every sum in the order of RKF45's threads (rhs_thread without TEAM), whose
// values it then returns bit for bit (one pass over all reactions: qq.chunk >=
// m.R).
template <bool INT, bool ORD = false>
static __device__ __noinline__ void team_rhs(const DevMech& m, const double* tab, double p, int y_o, int f_o,
                                             int bufs_o, int vp, RhsQ qq) {
  extern __shared__ __align__(16) double sm[];
  const double* y = sm + y_o;
  double* f = sm + f_o;
  TeamBufs b = carve_bufs(sm + bufs_o, m.S, sm + qq.off, 0, vp);
  Mix x;
  const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const int S = m.S, SG = species_groups(S);
  const bool in = team_species<ORD, INT>(m, p, y, b, x, tab);
  const double invrho = x.invrho;
  // every chunk: its rates of progress, then one fixed-order gather per
  // species, longest rows first so that the lanes of a warp do similar work
  // (one chunk when q holds all reactions)
  const int CH = qq.chunk;
  for (int base = 0;;) {
    const int cnt = m.R - base < CH ? m.R - base : CH;
    // last reactions first: the expensive ones (fall-off) then fill whole
    // warps, and the warp that is left partly empty has the cheapest
    if (INT && in) {
      for (int li = cnt - 1 - tid; li >= 0; li -= blockDim.x)
        team_reaction<false, INT, ORD>(m, m.rxn + base + li, x, b, tab, li, 0);
    } else {
      for (int li = cnt - 1 - tid; li >= 0; li -= blockDim.x)
        team_reaction<false, false, ORD>(m, m.rxn + base + li, x, b, tab, li, 0);
    }
    team_sync();
    const bool last = base + cnt >= m.R;
    for (int kk = tid; kk < S; kk += blockDim.x) {
      const int k = m.rsp[kk];
      const int32_t* ptr = ORD ? m.slot_ptr : m.csr_ptr;
      const CsrTerm* terms = ORD ? m.slot : m.csr;
      int e = ptr[k], e1 = ptr[k + 1];
      double w = 0.0;
      if (!ORD && CH < m.R) {
        const int c = base / CH;
        const int* cp = m.csr_cptr + k * (m.n_rhs_chunks + 1) + c;
        e = cp[0];
        e1 = cp[1];
        if (c) w = b.wd[k];
      }
      for (; e < e1; ++e) {
        const CsrTerm t = terms[e];
        w = fma(t.nu, b.q[t.rx - base], w);
      }
      b.wd[k] = w;
      if (last) f[1 + k] = w * (m.W[k] * invrho);
    }
    team_sync();
    if (last) break;
    base += CH;
  }
  // dT/dt by the last warp: its two species sums and the division.  Constant
  // volume: U/RT = H/RT - 1, cv/R = cp/R - 1.
  if (warp == nw - 1) {
    double cpm[4] = {0.0, 0.0, 0.0, 0.0}, hw[4] = {0.0, 0.0, 0.0, 0.0};
    const bool fold = b.vp == 64;
    const int ng = fold && SG > 2 ? 2 : SG;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q < SG) {
        const int k = 32 * q + lane;
        if (k < S) {
          double c = b.cpR[k], h = b.hRT[k];
          if (m.cv) {
            c -= 1.0;
            h -= 1.0;
          }
          const double yk = y[1 + k] * m.invW[k], w = b.wd[k];
          if (q >= 2 && fold) {
            cpm[q - 2] = fma(yk, c, cpm[q - 2]);
            hw[q - 2] = fma(h, w, hw[q - 2]);
          } else {
            cpm[q] = fma(yk, c, 0.0);
            hw[q] = fma(h, w, 0.0);
          }
        }
      }
    double sc, sh;
    if (ORD) {
      // lane 0 the heat capacity, lane 1 the enthalpy, both from one chain
      // (the factors side by side in the Gibbs arrays, free by now)
      for (int k = lane; k < S; k += 32) {
        b.Gp[k] = y[1 + k] * m.invW[k];
        b.Gm[k] = m.cv ? b.cpR[k] - 1.0 : b.cpR[k];
        if (m.cv) b.hRT[k] -= 1.0;
      }
      __syncwarp();
      const double* a0 = lane & 1 ? b.hRT : b.Gp;
      const double* a1 = lane & 1 ? b.wd : b.Gm;
      double s = 0.0;
      for (int k = 0; k < S; ++k) s = fma(a0[k], a1[k], s);
      sc = __shfl_sync(0xffffffffu, s, 0);
      sh = __shfl_sync(0xffffffffu, s, 1);
    } else if (ng <= 2) {
      const double v = warp_sum_pack4(cpm[0], cpm[1], hw[0], hw[1]);
      // lanes 0-15: cpm, 16-31: hw, both from one add
      const double s = v + __shfl_xor_sync(0xffffffffu, v, 8);
      sc = __shfl_sync(0xffffffffu, s, 0);
      sh = __shfl_sync(0xffffffffu, s, 16);
    } else {
      sc = warp_sum_groups(cpm, ng);
      sh = warp_sum_groups(hw, ng);
    }
    if (lane == 0) f[0] = -x.T * sh / (x.rho * sc);
  }
  team_sync();
}

// The right-hand side of a kernel: LAT kernels (four warps, at most 32 species)
// take the latency form for mechanisms of few reactions, whose rates q holds all.
template <bool INT, bool ORD, bool LAT>
__device__ __forceinline__ void team_rhs_any(const DevMech& m, const double* tab, double p, int y_o, int f_o,
                                             int bufs_o, int vp, RhsQ qq) {
  if (LAT && latency_form(m)) team_rhs_lat<ORD>(m, tab, p, y_o, f_o, bufs_o, qq.off);
  else team_rhs<INT, ORD>(m, tab, p, y_o, f_o, bufs_o, vp, qq);
}

// Analytic Jacobian J = df/d(T, Y) at constant p, written row-major into A
// (rows jt.ld apart), and into M too (rows ldm apart) unless that is NULL, and
// f(y) into f.  Derivation
// (chain rule through rho(T, Y) and [X](rho, Y); dlnK_c/dT = (sum nu H/RT -
// dnu)/T):
//   A_kj   = sum_i nu_ki dq_i/d[X_j] (sparse mass-action part and the
//            (eff - 1) corrections) + u_k (dense third-body part, u_k = sum nu_ki w_i),
//   E_k    = sum_i nu_ki D_i,  a_k = sum_i nu_ki dq_i/dT,
//   J[1+k][1+j] = (W_k (A_kj + u_k) + W_k Wbar (wdot_k - E_k)/rho) / W_j,
//   J[1+k][0]   = W_k (a_k + wdot_k / T) / rho,
//   J[0][1+j]   = -(T (rho cs_j - Wbar HE)/(rho cpm) + Tdot (cp_j/cpm - Wbar)) / W_j,
//   J[0][0]     = -(sum cp_k wdot_k + T sum H_k/RT a_k)/(rho cpm) - Tdot (dcpm/cpm - 1/T),
// with cs_j = sum_k H_k/RT (A_kj + u_k), HE = sum_k H_k/RT E_k, and heat
// capacities in units of R.  Constant volume (rho fixed; u_k, c_v in Eq.
// tdot): the Wbar and 1/T terms vanish, a_k is taken at fixed [X], and H/RT,
// cp/R become U/RT = H/RT - 1 and cv/R = cp/R - 1:
//   J[1+k][1+j] = W_k (A_kj + u_k) / W_j,   J[1+k][0] = W_k a_k / rho,
//   J[0][1+j]   = -(T cs_j / cvm + Tdot cv_j / cvm) / W_j,
//   J[0][0]     = -(sum cv_k wdot_k + T sum U_k/RT a_k)/(rho cvm) - Tdot dcpm/cvm.
// The species block is accumulated in A.  With A in device memory (where it
// stays in L2) the per-reaction values (b.q and on) may lie where M is: they
// are read for the last time before M is written, so that a team needs shared
// memory for the larger of the two only, and takes all reactions in one pass.
// Needs b.vp >= S (one species a lane in the sums).
// Bound by the FP64 unit: ck_jacobian on 8192 reactors of the 53-species
// mechanism 0.96 ms (1.59 with chunks of 64 reactions accumulated in shared
// memory and every sum taken by every warp); on 900 of the 111-species one
// 0.34 ms (0.64).
template <bool INT, bool LAT = false>
static __device__ void team_jacobian(const DevMech& m, const JacTab& jt, const double* tab, double p, const double* y,
                                     double* f, double* A, double* M, int ldm, TeamBufs b) {
  Mix x;
  const int S = m.S, lda = jt.ld, na = m.n * lda, SG = species_groups(S);
  const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const bool lat = LAT && latency_form(m);
  bool in = false;
  if (lat) team_species_lat<false, true>(m, p, y, b, x, tab, b.q, b.w);
  else in = team_species<false, INT>(m, p, y, b, x, tab);
  // chunk by chunk, every target (species-block entries and the per-species
  // sums wdot, a, E, u, whose arrays wd, aT, E, u are contiguous) adds its
  // fixed-order sum of terms; one thread per target, no conflicts, the
  // targets sorted by length so that a warp's lanes do similar work
  for (int c = 0; c < jt.n_chunks; ++c) {
    const int base = c * jt.chunk, cnt = m.R - base < jt.chunk ? m.R - base : jt.chunk;
    const int ft = m.first_typed > base ? m.first_typed - base : 0;
    if (lat) {
      for (int s = tid; s < lat_slots(cnt, m.first_typed); s += blockDim.x) {
        const int li = lat_reaction(s, m.first_typed);
        if (li >= 0) team_reaction<true, false, false, true>(m, m.rxn + li, x, b, tab, li, li - ft);
      }
    } else if (INT && in) {
      for (int li = cnt - 1 - tid; li >= 0; li -= blockDim.x)
        team_reaction<true, INT>(m, m.rxn + base + li, x, b, tab, li, li - ft);
    } else {
      for (int li = cnt - 1 - tid; li >= 0; li -= blockDim.x)
        team_reaction<true, false>(m, m.rxn + base + li, x, b, tab, li, li - ft);
    }
    team_sync();
    for (int e = jt.jc_ptr[c] + tid; e < jt.jc_ptr[c + 1]; e += blockDim.x) {
      const JcEntry h = jt.jc[e];
      double a = 0.0;
      if (c > 0) a = h.idx < na ? A[h.idx] : b.wd[h.idx - na];
      for (int t = h.beg; t < h.end; ++t) {
        const JcTerm ct = jt.jt[t];
        a = fma(ct.coef, b.q[ct.pidx], a);
      }
      if (h.idx < na) A[h.idx] = a;
      else b.wd[h.idx - na] = a;
    }
    team_sync();
  }
  // Constant volume: rho is fixed, so every term that comes from d rho/dT or
  // d rho/dY (cpf) drops out, and U/RT = H/RT - 1, cv/R = cp/R - 1 take the
  // places of H/RT and cp/R (cvf).  The contributions were pre-scaled by
  // W_k/W_j, so A holds A'_kj = W_k A_kj / W_j here.
  const double invrho = x.invrho;
  const double cvf = m.cv ? 1.0 : 0.0, cpf = 1.0 - cvf;
  double* eW = b.Gm;     // e_k / W_k, for the column sums
  double* dense = b.X;   // dense part of the species block, W_k u_k + W_k Wbar (wdot_k - E_k) / rho
  double* cs = b.Gp;
  for (int k = tid; k < S; k += blockDim.x) {
    f[1 + k] = b.wd[k] * (m.W[k] * invrho);
    eW[k] = (b.hRT[k] - cvf) * m.invW[k];
    dense[k] = m.W[k] * fma(cpf * x.Wbar * invrho, b.wd[k] - b.E[k], b.u[k]);
  }
  team_sync();
  // the last warp: the seven species sums (cpm, dcpm, hw, he, cw, ha, eu),
  // Tdot and 1 / cpm; the others: cs'_j = sum_k (e_k / W_k) A'_kj
  double* sums = b.red + SC_SUM;
  if (warp == nw - 1) {
    const double T2 = b.red[SC_T2], T3 = b.red[SC_T3];
    double sv = 0.0;  // lane q: sum q over the groups so far
#pragma unroll
    for (int g = 0; g < 4; ++g)
      if (g < SG) {
        const int k = 32 * g + lane;
        double v[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        if (k < S) {
          const double* a = m.thermo + k * TH_PER_SPECIES + (x.T < m.tmid[k] ? 0 : TH_STRIDE);
          const double yk = y[1 + k] * m.invW[k];
          const double e = b.hRT[k] - cvf, c = b.cpR[k] - cvf;
          v[0] = fma(yk, c, 0.0);
          v[1] = fma(yk, fma(4.0 * a[4], T3, fma(3.0 * a[3], T2, fma(2.0 * a[2], x.T, a[1]))), 0.0);
          v[2] = fma(e, b.wd[k], 0.0);
          v[3] = fma(b.hRT[k], b.E[k], 0.0);
          v[4] = fma(c, b.wd[k], 0.0);
          v[5] = fma(e, b.aT[k], 0.0);
          v[6] = fma(e, b.u[k], 0.0);
        }
        const double s = warp_sum_pack8(v);  // lane 4 q holds sum q
        sv = g == 0 ? s : sv + s;
      }
    const double cpm = __shfl_sync(0xffffffffu, sv, 0), hw = __shfl_sync(0xffffffffu, sv, 8);
    const double Tdot = -x.T * hw / (x.rho * cpm);
    const double inv_cpm = rcp_rn(cpm);
    if ((lane & 3) == 0 && lane < 28) sums[lane >> 2] = sv;
    if (lane == 0) {
      b.red[SC_TDOT] = Tdot;
      b.red[SC_ICPM] = inv_cpm;
    }
  }
  // (a team of one warp does both; otherwise the column sums start at warp 0)
  for (int g = warp; g < SG; g += nw) {
    const int j = 32 * g + lane;
    if (j < S) {
      double s = 0.0;
      const double* a = A + lda + 1 + j;
#pragma unroll 8
      for (int k = 0; k < S; ++k) s = fma(eW[k], a[k * lda], s);
      cs[j] = s;
    }
  }
  team_sync();
  const double dcpm = sums[1], he = sums[3], cw = sums[4], ha = sums[5], eu = sums[6];
  const double Tdot = b.red[SC_TDOT], inv_cpm = b.red[SC_ICPM];
  // species block (J_kj = A'_kj + dense_k / W_j), entries e = k S + j, (k, j)
  // advanced without dividing by the runtime S
  {
    const int P = blockDim.x, dk = P / S, dj = P - (P / S) * S;
    int k = tid / S, j = tid - k * S;
    for (; k < S;) {
      double* a = A + (1 + k) * lda + 1 + j;
      const double v = fma(dense[k], m.invW[j], *a);
      *a = v;
      if (M) M[(1 + k) * ldm + 1 + j] = v;
      k += dk;
      j += dj;
      if (j >= S) {
        j -= S;
        ++k;
      }
    }
  }
  // temperature column and row (each product rounded where it is written)
  for (int k = tid; k < S; k += blockDim.x) {
    const double v = m.W[k] * invrho * fma(cpf * b.wd[k], x.invT, b.aT[k]);
    A[(1 + k) * lda] = v;
    if (M) M[(1 + k) * ldm] = v;
  }
  const double inv_rc = invrho * inv_cpm;
  for (int j = tid; j < S; j += blockDim.x) {
    // cs_j = sum_k e_k (A_kj + u_k) = W_j sum_k (e_k / W_k) A'_kj + sum_k e_k u_k
    const double csj = fma(m.W[j], cs[j], eu);
    const double cW = __dmul_rn(cpf, x.Wbar);
    const double d0 = fma(x.rho, csj, -__dmul_rn(cW, he));
    const double tt = fma(__dmul_rn(x.T, d0), inv_rc, __dmul_rn(Tdot, fma(b.cpR[j] - cvf, inv_cpm, -cW)));
    const double v = -tt * m.invW[j];
    A[1 + j] = v;
    if (M) M[1 + j] = v;
  }
  if (tid == 0) {
    const double v = fma(-fma(x.T, ha, cw), inv_rc, -__dmul_rn(Tdot, fma(dcpm, inv_cpm, -cpf * x.invT)));
    A[0] = v;
    if (M) M[0] = v;
    f[0] = Tdot;
  }
  team_sync();
}

// LU with partial pivoting of the n x n row-major matrix A (shared memory,
// n <= 144, rows ld = lu_ld(n) apart) by the whole team, in place.  An FP64 instruction costs a full
// warp slot of a pipe that takes 64 cycles a slot, while shared memory has
// bandwidth to spare beside it (an update moves 3 loads and a store per
// slot), so the trailing matrix stays in shared memory and its elements are
// dealt to the lanes one by one, as a flat list: a pivot with m rows below it
// costs ceil(m^2 / 32) slots, with no lanes lost to the edges of a tile, and
// the team keeps no tile in registers (which lets more warps reside).
// Rows are never moved: rows k.. of the permuted matrix are listed, with
// their multipliers, in a row table (LuRow), rebuilt for every pivot.
// One barrier a pivot: while the other warps update columns k + 2.. with
// pivot k, one warp (a different one each time) updates column k + 1, picks
// pivot k + 1 in it and forms its multipliers and row table (two tables, used
// in turn).  Every element receives its updates in pivot order, so the
// factors do not depend on how the elements are dealt.
// GB300, 4096 matrices of 54: 502 us a factorization of all (838 with register
// tiles and two barriers a pivot; the FP64 unit's floor is about 360), 1.72 k
// FP64 warp instructions a matrix (2.80 k); 900 of 112: 959 us (1539).
// Pivot: the largest magnitude of rows i >= k, ties to the smallest row
// (magnitudes compared as integers: the bit pattern of |v| orders like |v|,
// NaN above +inf).
// On return rof[i] holds row i of PA as (its offset in A << 8) | row, A the
// unit lower factor below the diagonal and the upper factor on and above it
// (row i of them at offset rof[i] >> 8), invd[k] = 1 / U_kk.  PRE: the strict
// upper triangle is stored divided by its diagonal, so that back
// substitution needs no division.  lpiv (may be NULL) receives the row that
// pivot k was swapped with (LAPACK order).  Returns 0, or k + 1 when pivot k
// is zero or not finite (the same in every thread; A then holds the matrix as
// updated by the pivots before k).
// lr: 2 n entries of scratch, flag: two ints of shared memory.  Pivot k raises
// flag[k & 1]: the panel of pivot k + 1 may run while a slower warp has yet to
// read pivot k's, behind the barrier that both have passed, and a flag that it
// saw too early would take that warp out of the loop one barrier before its
// team.
template <class F>
struct __align__(2 * sizeof(F)) LuRow {
  F l;      // multiplier
  int pk;   // (offset << 8) | row of A
};

// Bits of |v| as an unsigned integer (orders like |v|; NaN above +inf).
__device__ __forceinline__ unsigned long long abs_key(double v) {
  return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffULL;
}
__device__ __forceinline__ unsigned long long abs_key(float v) {
  return (unsigned long long)((unsigned)__float_as_int(v) & 0x7fffffffu) << 32;
}
__device__ __forceinline__ unsigned long long inf_key(double) { return 0x7ff0000000000000ULL; }
__device__ __forceinline__ unsigned long long inf_key(float) { return 0x7f80000000000000ULL; }

constexpr int LU_MAX_N = 144;

// Pivot k, by one warp: column k updated with pivot k - 1, the pivot of rows
// k.., and the multipliers and row order of the rows below it.
template <class F>
__device__ __forceinline__ void lu_panel(F* A, int n, int k, int* rof, int* lpiv, F* invd, LuRow<F>* lr, int* flag) {
  constexpr int Q = (LU_MAX_N + 31) / 32;
  const int lane = threadIdx.x & 31;
  const LuRow<F>* prev = lr + ((k + 1) & 1) * n;
  LuRow<F>* next = lr + (k & 1) * n;
  const F u = k > 0 ? A[(rof[k > 0 ? k - 1 : 0] >> 8) + k] : F(0);
  F v[Q];
  int pk[Q];
  unsigned long long best = 0;
  F bv = F(0);
  int bi = n, bpk = 0;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int i = k + lane + 32 * q;
    v[q] = F(0);
    pk[q] = 0;
    if (k + 32 * q < n) {  // warp-uniform
      if (i < n) {
        const LuRow<F> r = prev[i];
        pk[q] = r.pk;
        v[q] = A[(r.pk >> 8) + k];
        if (k > 0) v[q] = fma(-r.l, u, v[q]);
        const unsigned long long key = abs_key(v[q]);
        if (key > best) {
          best = key;
          bv = v[q];
          bi = i;
          bpk = r.pk;
        }
      }
    }
  }
  const unsigned hi = (unsigned)(best >> 32);
  const unsigned H = __reduce_max_sync(0xffffffffu, hi);
  unsigned L = 0;
  if (sizeof(F) == 8) L = __reduce_max_sync(0xffffffffu, hi == H ? (unsigned)best : 0u);
  const bool mine = hi == H && (sizeof(F) < 8 || (unsigned)best == L);
  const int p = (int)__reduce_min_sync(0xffffffffu, mine ? (unsigned)bi : (unsigned)n);
  const unsigned long long top = ((unsigned long long)H << 32) | L;
  if (p >= n || top == 0 || top >= inf_key(F(0))) {
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int i = k + lane + 32 * q;
      if (i < n) {
        A[(pk[q] >> 8) + k] = v[q];
        rof[i] = pk[q];  // the row order as it stands
      }
    }
    if (lane == 0) flag[k & 1] = k + 1;
    return;
  }
  const int from = (p - k) & 31;
  bv = __shfl_sync(0xffffffffu, bv, from);
  bpk = __shfl_sync(0xffffffffu, bpk, from);
  const F vk = __shfl_sync(0xffffffffu, v[0], 0);
  const int pkk = __shfl_sync(0xffffffffu, pk[0], 0);
  const F ip = rcp_int(bv);
  if (lane == 0) {
    rof[k] = bpk;
    A[(bpk >> 8) + k] = bv;
    invd[k] = ip;
    if (lpiv) lpiv[k] = p;
  }
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int i = k + lane + 32 * q;
    if (k + 32 * q < n) {
      // row p takes row k's entry
      LuRow<F> r;
      r.l = (i == p ? vk : v[q]) * ip;
      r.pk = i == p ? pkk : pk[q];
      if (i > k && i < n) {
        next[i] = r;
        A[(r.pk >> 8) + k] = r.l;
      }
    }
  }
}

// Element e of a list of rows of c elements: its row, for e < 2^15, c <= 144
// (rc = 1 / c in FP32: (e + 1/2) / c is at least 1 / (2 c) away from an
// integer, far more than its rounding error of 2^-22 e / c).
__device__ __forceinline__ int flat_row(int e, float rc) { return (int)(((float)e + 0.5f) * rc); }

// Rows i0, i0 + step, .. of the m x c trailing matrix at A2, updated with the
// pivot row U and the multipliers in R.
template <class F>
__device__ __forceinline__ void lu_rows(F* A2, const F* U, const LuRow<F>* R, int m, int c, int i0, int step) {
  constexpr int Q = (LU_MAX_N + 31) / 32;
  const int lane = threadIdx.x & 31;
  F u[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) u[q] = lane + 32 * q < c ? U[lane + 32 * q] : F(0);
  for (int i = i0; i < m; i += 2 * step) {
    const bool two = i + step < m;
    const LuRow<F> r0 = R[i], r1 = R[two ? i + step : i];
    F* a0 = A2 + (r0.pk >> 8) + lane;
    F* a1 = A2 + (r1.pk >> 8) + lane;
    F v0[Q], v1[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const bool in = lane + 32 * q < c;
      v0[q] = in ? a0[32 * q] : F(0);
      v1[q] = in ? a1[32 * q] : F(0);
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      if (lane + 32 * q < c) {
        a0[32 * q] = fma(-r0.l, u[q], v0[q]);
        if (two) a1[32 * q] = fma(-r1.l, u[q], v1[q]);
      }
    }
  }
}

template <bool PRE, class F>
__device__ __forceinline__ int lu_flat(F* A, int n, int* rof, int* lpiv, F* invd, LuRow<F>* lr, int* flag) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  for (int i = tid; i < n; i += blockDim.x) {
    lr[n + i].pk = (i * lu_ld(n)) << 8 | i;
    if (lpiv) lpiv[i] = i;
  }
  if (tid < 2) flag[tid] = 0;
  team_sync();
  if (warp == 0) lu_panel(A, n, 0, rof, lpiv, invd, lr, flag);
  team_sync();
  if (flag[0]) return flag[0];
  constexpr int C0 = 10;  // a panel costs its warp about as much as this many updates of 32 elements
  int pw = 1 % nw;        // the warp of the next panel
  for (int k = 0; k + 1 < n; ++k) {
    const int m = n - 1 - k, mc = m - 1, E = m * mc, NG = (E + 31) >> 5;
    if constexpr (sizeof(F) == 4) {
      // FP32 (the precision form): the arithmetic is cheap and the index work
      // of the flat list would set the pace, so a lane keeps its columns and
      // the other warps take rows in turn
      if (warp == pw) lu_panel(A, n, k + 1, rof, lpiv, invd, lr, flag);
      if (warp != pw || nw == 1)
        lu_rows(A + k + 2, A + (rof[k] >> 8) + k + 2, lr + (k & 1) * n + k + 1, m, mc,
                nw == 1 ? 0 : (warp > pw ? warp - pw - 1 : warp - pw - 1 + nw), nw == 1 ? 1 : nw - 1);
      if (++pw == nw) pw = 0;
      team_sync();
      if (flag[(k + 1) & 1]) return flag[(k + 1) & 1];
      continue;
    }
    // groups of 32 elements: the panel's warp takes the last gp, the others
    // share the rest
    int gp = NG, g0 = 0, gs = 1, g1 = NG;
    if (nw > 1) {
      const int per = (NG + C0 + nw - 1) / nw;
      gp = per > C0 ? per - C0 : 0;
      if (warp == pw) {
        g0 = NG - gp;
      } else {
        g0 = warp - pw - 1;
        if (g0 < 0) g0 += nw;
        gs = nw - 1;
        g1 = NG - gp;
      }
    }
    if (warp == pw) lu_panel(A, n, k + 1, rof, lpiv, invd, lr, flag);
    const LuRow<F>* R = lr + (k & 1) * n + k + 1;
    const F* U = A + (rof[k] >> 8) + k + 2;
    F* A2 = A + k + 2;
    const float rc = 1.0f / (float)(mc > 0 ? mc : 1);
    int g = g0;
    for (; g + 3 * gs < g1; g += 4 * gs) {
      F l[4], u[4], a[4];
      int o[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int e0 = 32 * (g + t * gs) + lane, e = e0 < E ? e0 : E - 1;
        const int i = flat_row(e, rc), j = e - i * mc;
        const LuRow<F> r = R[i];
        l[t] = r.l;
        u[t] = U[j];
        o[t] = (r.pk >> 8) + j;
        a[t] = A2[o[t]];
        if (e0 >= E) o[t] = -1;
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const F w = fma(-l[t], u[t], a[t]);
        if (o[t] >= 0) A2[o[t]] = w;
      }
    }
    for (; g < g1; g += gs) {
      const int e = 32 * g + lane;
      if (e < E) {
        const int i = flat_row(e, rc), j = e - i * mc;
        const LuRow<F> r = R[i];
        F* a = A2 + (r.pk >> 8) + j;
        *a = fma(-r.l, U[j], *a);
      }
    }
    if (++pw == nw) pw = 0;
    team_sync();
    if (flag[(k + 1) & 1]) return flag[(k + 1) & 1];
  }
  if (PRE) {
    // rows r and n - 2 - r of the strict upper triangle have n elements together
    const int E = n * (n - 1) / 2;
    const float rc = 1.0f / (float)n;
    for (int e = tid; e < E; e += blockDim.x) {
      const int r = flat_row(e, rc), c = e - r * n, m = n - 1 - r;
      const int i = c < m ? r : n - 2 - r, j = c < m ? r + 1 + c : n - 1 - r + (c - m);
      F* a = A + (rof[i] >> 8) + j;
      *a = *a * invd[i];
    }
    team_sync();
  }
  return 0;
}

// Solve (LU) x = b in place with one warp (b in shared memory).  Must be
// called by all 32 lanes of one warp; the caller orders it against the rest
// of the CTA with a barrier.  Blocked by 32 rows: the dependence of a block on
// earlier blocks is a matrix-vector product (one row per lane, four partial
// sums in a fixed order), the diagonal block a substitution whose solved
// value is broadcast by a shuffle.
// PRE: the factors come from lu_flat<true> (rows listed in its row table rof,
// passed as piv: gather by it, U pre-divided by its diagonal); else rows in
// order, lu_ld(n) apart, and piv[k] the row swapped with row k.
template <bool PRE = false, class F>
__device__ __forceinline__ void warp_lu_solve(const F* A, int n, const int* piv, const F* invd, F* b) {
  const int lane = threadIdx.x & 31;
  if (PRE) {
    constexpr int MAXR = 5;  // n <= 160 (the team kernels take n <= 144)
    F g[MAXR];
#pragma unroll
    for (int q = 0; q < MAXR; ++q) {
      const int i = lane + 32 * q;
      g[q] = i < n ? b[piv[i] & 255] : F(0);
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < MAXR; ++q) {
      const int i = lane + 32 * q;
      if (i < n) b[i] = g[q];
    }
  } else if (lane == 0) {
    for (int k = 0; k < n; ++k) {
      const int p = piv[k];
      if (p != k) {
        const F t = b[k];
        b[k] = b[p];
        b[p] = t;
      }
    }
  }
  __syncwarp();
  // forward substitution with the unit lower triangle
  for (int B0 = 0; B0 < n; B0 += 32) {
    const int i = B0 + lane;
    const bool act = i < n;
    F s0 = act ? b[i] : F(0), s1 = F(0), s2 = F(0), s3 = F(0);
    const F* Li = A + (PRE ? (act ? piv[i] >> 8 : 0) : (act ? i : 0) * lu_ld(n));
    if (act) {
      int j = 0;
      for (; j + 4 <= B0; j += 4) {
        s0 = fma(-Li[j], b[j], s0);
        s1 = fma(-Li[j + 1], b[j + 1], s1);
        s2 = fma(-Li[j + 2], b[j + 2], s2);
        s3 = fma(-Li[j + 3], b[j + 3], s3);
      }
      for (; j < B0; ++j) s0 = fma(-Li[j], b[j], s0);
    }
    F s = (s0 + s1) + (s2 + s3);
    const int m = min(32, n - B0);
    for (int jj = 0; jj < m; ++jj) {
      const F yj = __shfl_sync(0xffffffffu, s, jj);
      if (act && lane > jj) s = fma(-Li[B0 + jj], yj, s);
    }
    if (act) b[i] = s;
    __syncwarp();
  }
  // back substitution with U
  for (int B1 = ((n - 1) / 32) * 32; B1 >= 0; B1 -= 32) {
    const int i = B1 + lane;
    const bool act = i < n;
    const int m = min(32, n - B1);
    F s0 = act ? (PRE ? b[i] * invd[i] : b[i]) : F(0), s1 = F(0), s2 = F(0), s3 = F(0);
    const F* Ui = A + (PRE ? (act ? piv[i] >> 8 : 0) : (act ? i : 0) * lu_ld(n));
    if (act) {
      int j = B1 + 32;
      for (; j + 4 <= n; j += 4) {
        s0 = fma(-Ui[j], b[j], s0);
        s1 = fma(-Ui[j + 1], b[j + 1], s1);
        s2 = fma(-Ui[j + 2], b[j + 2], s2);
        s3 = fma(-Ui[j + 3], b[j + 3], s3);
      }
      for (; j < n; ++j) s0 = fma(-Ui[j], b[j], s0);
    }
    F s = (s0 + s1) + (s2 + s3);
    for (int jj = m - 1; jj >= 0; --jj) {
      if (!PRE && lane == jj) s *= invd[i];
      const F xj = __shfl_sync(0xffffffffu, s, jj);
      if (act && lane < jj) s = fma(-Ui[B1 + jj], xj, s);
    }
    if (act) b[i] = s;
    __syncwarp();
  }
}

// lu_flat<true> and its solve out of line (one copy of each in a kernel that
// calls them often), with their arrays by offset (doubles; b_o in elements) in
// the CTA's dynamic shared memory so that they still address it directly.
template <class F>
static __device__ __noinline__ int team_lu(int a_o, int n, int rof_o, int invd_o, int lr_o, int flag_o) {
  extern __shared__ __align__(16) double sm[];
  return lu_flat<true>(reinterpret_cast<F*>(sm + a_o), n, reinterpret_cast<int*>(sm + rof_o), nullptr,
                       reinterpret_cast<F*>(sm + invd_o), reinterpret_cast<LuRow<F>*>(sm + lr_o),
                       reinterpret_cast<int*>(sm + flag_o));
}
template <class F>
static __device__ __noinline__ void warp_solve(int a_o, int n, int rof_o, int invd_o, int b_o) {
  extern __shared__ __align__(16) double sm[];
  warp_lu_solve<true>(reinterpret_cast<const F*>(sm + a_o), n, reinterpret_cast<const int*>(sm + rof_o),
                      reinterpret_cast<const F*>(sm + invd_o), reinterpret_cast<F*>(sm) + b_o);
}

}  // namespace ck
