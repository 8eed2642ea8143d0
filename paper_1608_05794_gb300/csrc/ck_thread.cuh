// Thread-per-reactor right-hand side ("shallow" vectorisation, Sec. 4 of
// the paper: one ODE system per SIMT lane).  Every lane walks the same
// reaction list, so table reads are uniform (broadcast) and the only
// divergence is the per-species choice of NASA-7 range (Sec. 4, "Select").
#pragma once
#include "ck_common.cuh"

namespace ck {

// Tables as seen by one kernel: shared memory when staged, else global.
struct MechView {
  int S, R;
  const RxnRec* rx;
  const double* th;
  const double* tmid;
  const double* W;
  const double* invW;
  const int16_t* eff_sp;
  const double* eff_m1;
  const double* tab;  // 2^(j/256), j = 0..255
  const double* revp; // explicit reverse rows: log2 A_r, beta_r, Ea_r / (R ln 2)
  int cv;             // 1: constant volume (p is the density)
};

// The reaction loop of rhs_thread: wd_k += nu q of every reaction, in order.
// INT: the products of concentrations and of Gibbs factors in integer
// arithmetic, beside the FP64 unit (see mul_int).  FEW: the powers of R T/p0 formed
// where they are used, for a kernel short of registers (RKF45 on 53 species
// 323 -> 313 ms; the right-hand side alone is 3 to 5 % faster with the four kept).
template <bool INT, bool FEW>
__device__ __forceinline__ void rates_thread(const MechView& m, double T, double invT, double log2T, double Ctot,
                                             const double* X, const double* G, const double* Gm, double* wd) {
  const double up = T * R_OVER_P0, up2 = up * up, dw = invT * P0_OVER_R, dw2 = dw * dw;
  for (int i = 0; i < m.R; ++i) {
    const RxnRec& r = m.rx[i];
    const double l2kf = fma(-r.EoR2, invT, fma(r.beta, log2T, r.lA2));
    const double kf = ck_exp2(l2kf, m.tab);
    double fwd = X[r.sp[0]];
    if (r.nreac > 1) fwd = mul_sel<INT>(fwd, X[r.sp[1]]);
    if (r.nreac > 2) fwd = mul_sel<INT>(fwd, X[r.sp[2]]);
    double net = kf * fwd;
    if (r.rev == 2) {
      const double* ra = m.revp + 3 * r.rev_ix;
      const double kr = ck_exp2(fma(-ra[2], invT, fma(ra[1], log2T, ra[0])), m.tab);
      double rv = X[r.sp[3]];
      if (r.nprod > 1) rv = mul_sel<INT>(rv, X[r.sp[4]]);
      if (r.nprod > 2) rv = mul_sel<INT>(rv, X[r.sp[5]]);
      net = fma(-kr, rv, net);
    } else if (r.rev) {
      const int dn = r.dnu;
      const double q = FEW ? rt_over_p0_pow(dn, T, invT)
                           : dn >= 0 ? (dn == 0 ? 1.0 : (dn == 1 ? up : up2)) : (dn == -1 ? dw : dw2);
      double kci = mul_sel<INT>(q, G[r.sp[0]]);
      kci = mul_sel<INT>(kci, Gm[r.sp[3]]);
      if (r.nreac > 1) kci = mul_sel<INT>(kci, G[r.sp[1]]);
      if (r.nprod > 1) kci = mul_sel<INT>(kci, Gm[r.sp[4]]);
      if (r.nreac > 2) kci = mul_sel<INT>(kci, G[r.sp[2]]);
      if (r.nprod > 2) kci = mul_sel<INT>(kci, Gm[r.sp[5]]);
      const double kr = kf * kci;
      double rv = X[r.sp[3]];
      if (r.nprod > 1) rv = mul_sel<INT>(rv, X[r.sp[4]]);
      if (r.nprod > 2) rv = mul_sel<INT>(rv, X[r.sp[5]]);
      net = fma(-kr, rv, net);
    }
    double q = net;
    if (r.type) {
      double M = Ctot;
      for (int e = r.eff_beg; e < r.eff_beg + r.eff_cnt; ++e) M = fma(m.eff_m1[e], X[m.eff_sp[e]], M);
      if (r.type == 1) {
        q = M * net;
      } else {
        const double l2k0 = fma(-r.E0oR2, invT, fma(r.beta0, log2T, r.lA02));
        const double Pr = ck_exp2(l2k0 - l2kf, m.tab) * M;
        q = net * (Pr / (1.0 + Pr));
      }
    }
    wd[r.sp[0]] -= q;
    if (r.nreac > 1) wd[r.sp[1]] -= q;
    if (r.nreac > 2) wd[r.sp[2]] -= q;
    wd[r.sp[3]] += q;
    if (r.nprod > 1) wd[r.sp[4]] += q;
    if (r.nprod > 2) wd[r.sp[5]] += q;
  }
}

// f = (dT/dt, dY_k/dt) at state y (Eqs. ydot, tdot, wdot, kfor, krev, kc,
// tfits).  y and f are strided (element k at y[k*ys]); X and wd are per-lane
// scratch of S doubles, G of 2S (the species factors 2^(g_k), 2^(-g_k)).
//   rho = p Wbar / (R T), [X_k] = rho Y_k / W_k,
//   k_f = 2^(log2 A + beta log2 T - Ea/(R T ln 2)),
//   1/K_c = (R T/p0)^dnu prod_reactants 2^(g_j) prod_products 2^(-g_j), g_j = (S/R - H/RT)_j / ln 2,
//   k_r = k_f / K_c,
//   c = 1, [M], or P_r/(1+P_r) with P_r = 2^(log2 k0 - log2 k_inf) [M],
//   q = c (k_f prod [X]^nu' - k_r prod [X]^nu''),  wdot_k = sum (nu'' - nu') q,
//   dY_k/dt = wdot_k W_k / rho, dT/dt = -T sum_k (H_k/RT) wdot_k / (rho sum_k Y_k (cp_k/R)/W_k).
// Explicit reverse rows: k_r = 2^(log2 A_r + beta_r log2 T - Ea_r/(R T ln 2)).
// Constant volume (Sec. 3): rho = p (the parameter is the density) and
// H/RT -> U/RT = H/RT - 1, cp/R -> cv/R = cp/R - 1 in dT/dt.
template <bool INT, bool FEW = false>
__device__ __forceinline__ void rhs_thread(const MechView& m, double p, const double* y, int ys,
                                           double* f, int fs, double* X, double* G, double* wd) {
  const int S = m.S;
  const double T = y[0];
  const double invT = __drcp_rn(T);
  const double lnT = log(T);
  const double log2T = lnT * INV_LN2;
  const double T2 = T * T, T3 = T2 * T, T4 = T3 * T;
  double sumYW = 0.0;
  for (int k = 0; k < S; ++k) sumYW = fma(y[(1 + k) * ys], m.invW[k], sumYW);
  const double rho = m.cv ? p : p / (R_GAS * T * sumYW);
  double Ctot = 0.0;
  bool in = INT && temp_in_range(T);
  for (int k = 0; k < S; ++k) {
    const double xk = rho * (y[(1 + k) * ys] * m.invW[k]);
    X[k] = xk;
    Ctot += xk;
    if (INT) in &= conc_in_range(xk);
    const double* a = m.th + k * TH_PER_SPECIES + (T < m.tmid[k] ? 0 : TH_STRIDE);
    double g = fma(a[11], lnT, a[12]);
    g = fma(a[13], T, g);
    g = fma(a[14], T2, g);
    g = fma(a[15], T3, g);
    g = fma(a[16], T4, g);
    g = fma(a[17], invT, g);
    if (INT) in &= gibbs_in_range(g);
    ck_exp2_pm(g, m.tab, G[k], G[S + k]);
    wd[k] = 0.0;
  }
  const double* Gm = G + S;
  if constexpr (INT) {
    if (__all_sync(__activemask(), in)) rates_thread<true, FEW>(m, T, invT, log2T, Ctot, X, G, Gm, wd);
    else rates_thread<false, FEW>(m, T, invT, log2T, Ctot, X, G, Gm, wd);
  } else {
    rates_thread<false, FEW>(m, T, invT, log2T, Ctot, X, G, Gm, wd);
  }
  const double invrho = __drcp_rn(rho);
  const double cvf = m.cv ? 1.0 : 0.0;
  double cpm = 0.0, hw = 0.0;
  for (int k = 0; k < S; ++k) {
    const double* a = m.th + k * TH_PER_SPECIES + (T < m.tmid[k] ? 0 : TH_STRIDE);
    double cp = fma(a[4], T4, fma(a[3], T3, fma(a[2], T2, fma(a[1], T, a[0])))) - cvf;
    double h = fma(a[10], invT, fma(a[9], T4, fma(a[8], T3, fma(a[7], T2, fma(a[6], T, a[5]))))) - cvf;
    const double w = wd[k];
    cpm = fma(y[(1 + k) * ys] * m.invW[k], cp, cpm);
    hw = fma(h, w, hw);
    f[(1 + k) * fs] = w * (m.W[k] * invrho);
  }
  f[0] = -T * hw / (rho * cpm);
}

}  // namespace ck
