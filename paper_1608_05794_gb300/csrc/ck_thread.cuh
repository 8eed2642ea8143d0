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

struct Two {  // two sums side by side
  double a, b;
};
__device__ __forceinline__ Two operator+(const Two& x, const Two& y) { return {x.a + y.a, x.b + y.b}; }

// Sum of value(k) over the S species as a team takes it (warp_sum_groups: the
// butterfly tree of each 32 species, these one after another).  A group of n is
// walked in bit-reversed order, in which the tree needs one partial sum a level;
// `half` is the tree's widest stride below n.
template <class V, class F>
__device__ __forceinline__ V tree_sum(int S, F value) {
  V sum{};
  for (int g = 0; g < S; g += 32) {
    const int n = S - g < 32 ? S - g : 32;
    const int bits = n > 2 ? 31 - __clz(n - 1) : 0, half = 1 << bits;
    V s1{}, s2{}, s3{}, s4{}, v{};
#pragma unroll 1
    for (int i = 0; i < half; ++i) {
      const int k = bits ? (int)(__brev((unsigned)i) >> (32 - bits)) : 0;
      v = value(g + k);
      if (k + half < n) v = v + value(g + k + half);
      if (i & 1) {
        v = s1 + v;
        if (i & 2) {
          v = s2 + v;
          if (i & 4) {
            v = s3 + v;
            if (i & 8) v = s4 + v;
            else s4 = v;
          } else {
            s3 = v;
          }
        } else {
          s2 = v;
        }
      } else {
        s1 = v;
      }
    }
    sum = g ? sum + v : v;
  }
  return sum;
}

// The reaction loop of rhs_thread: wd_k += nu q of every reaction, in order.
// INT: the products of concentrations and of Gibbs factors in integer
// arithmetic, beside the FP64 unit (see mul_int).  TEAM: see rhs_thread; without
// it, also, the powers of R T/p0 formed where they are used, for a kernel short
// of registers.  WHOLE: a record's slots and kinds in two vector loads, taken apart in
// registers, instead of loads that wait for each other: the right-hand side of 53
// species 3050 -> 2960 us on 131072 reactors, RKF45 on 2000 325 -> 274 ms; the small
// mechanisms' RKF45 lacks the registers (1000 fixed steps of 100000 reactors 1.60 ->
// 1.71 s).
template <bool INT, bool TEAM, bool WHOLE>
__device__ __forceinline__ void rates_thread(const MechView& m, double T, double invT, double log2T, double Ctot,
                                             const double* X, const double* G, const double* Gm, double* wd) {
  const double up = T * R_OVER_P0, up2 = up * up, dw = invT * P0_OVER_R, dw2 = dw * dw;
  for (int i = 0; i < m.R; ++i) {
    const RxnRec& r = m.rx[i];
    int sp[6];
    int type, rev, dnu, nreac, nprod, repeats;
    if (WHOLE) {
      const uint4 h = *reinterpret_cast<const uint4*>(r.sp);
      const uint32_t g = *reinterpret_cast<const uint32_t*>(&r.nprod);
      sp[0] = h.x & 0xffff, sp[1] = h.x >> 16, sp[2] = h.y & 0xffff;
      sp[3] = h.y >> 16, sp[4] = h.z & 0xffff, sp[5] = h.z >> 16;
      type = h.w & 255, rev = h.w >> 8 & 255, dnu = (int8_t)(h.w >> 16), nreac = h.w >> 24;
      nprod = g & 255, repeats = g >> 8 & 255;
    } else {
      type = r.type, rev = r.rev, dnu = r.dnu, nreac = r.nreac, nprod = r.nprod, repeats = r.repeats;
    }
    auto slot = [&](int q) { return WHOLE ? sp[q] : (int)r.sp[q]; };
    const double l2kf = fma(-r.EoR2, invT, fma(r.beta, log2T, r.lA2));
    const double kf = ck_exp2(l2kf, m.tab);
    double fwd = X[slot(0)];
    if (nreac > 1) fwd = mul_sel<INT>(fwd, X[slot(1)]);
    if (nreac > 2) fwd = mul_sel<INT>(fwd, X[slot(2)]);
    double net = kf * fwd;
    if (rev == 2) {
      const double* ra = m.revp + 3 * r.rev_ix;
      const double kr = ck_exp2(fma(-ra[2], invT, fma(ra[1], log2T, ra[0])), m.tab);
      double rv = X[slot(3)];
      if (nprod > 1) rv = mul_sel<INT>(rv, X[slot(4)]);
      if (nprod > 2) rv = mul_sel<INT>(rv, X[slot(5)]);
      net = fma(-kr, rv, net);
    } else if (rev) {
      const double q = !TEAM ? rt_over_p0_pow(dnu, T, invT)
                             : dnu >= 0 ? (dnu == 0 ? 1.0 : (dnu == 1 ? up : up2)) : (dnu == -1 ? dw : dw2);
      double kci = mul_sel<INT>(q, G[slot(0)]);
      kci = mul_sel<INT>(kci, Gm[slot(3)]);
      if (nreac > 1) kci = mul_sel<INT>(kci, G[slot(1)]);
      if (nprod > 1) kci = mul_sel<INT>(kci, Gm[slot(4)]);
      if (nreac > 2) kci = mul_sel<INT>(kci, G[slot(2)]);
      if (nprod > 2) kci = mul_sel<INT>(kci, Gm[slot(5)]);
      const double kr = kf * kci;
      double rv = X[slot(3)];
      if (nprod > 1) rv = mul_sel<INT>(rv, X[slot(4)]);
      if (nprod > 2) rv = mul_sel<INT>(rv, X[slot(5)]);
      net = fma(-kr, rv, net);
    }
    double q = net;
    if (type) {
      double M = Ctot;
      for (int e = r.eff_beg; e < r.eff_beg + r.eff_cnt; ++e) M = fma(m.eff_m1[e], X[m.eff_sp[e]], M);
      if (type == 1) {
        q = M * net;
      } else {
        const double l2k0 = fma(-r.E0oR2, invT, fma(r.beta0, log2T, r.lA02));
        const double Pr = __dmul_rn(ck_exp2(l2k0 - l2kf, m.tab), M);
        q = net * (TEAM ? Pr * __drcp_rn(__dadd_rn(1.0, Pr)) : Pr / __dadd_rn(1.0, Pr));
      }
    }
    if (TEAM && repeats) {  // a species in several slots: its net coefficient at once
      auto add = [&](int k, int nu) {
        if (nu == 0) return;
        const int a = nu < 0 ? -nu : nu;  // 1.0, 2.0 or 3.0 and the sign
        const int hi = (a == 1 ? 0x3ff00000 : (a == 2 ? 0x40000000 : 0x40080000)) | (nu & (int)0x80000000);
        wd[k] = fma(__hiloint2double(hi, 0), q, wd[k]);
      };
      const uint32_t rn = REP_NET >> 6 * (repeats & 7), pn = REP_NET >> 6 * (repeats >> 3 & 7);
      if (repeats & REP_BOTH_SIDES) {
        // (rare: how often the species of slot k is on the other side, less)
        auto on = [&](int k, int from, int n) {
          int c = slot(from) == k;
          if (n > 1) c += slot(from + 1) == k;
          if (n > 2) c += slot(from + 2) == k;
          return c;
        };
        if (rn & 3) add(slot(0), on(slot(0), 3, nprod) - (int)(rn & 3));
        if (nreac > 1 && (rn >> 2 & 3)) add(slot(1), on(slot(1), 3, nprod) - (int)(rn >> 2 & 3));
        if (nreac > 2 && (rn >> 4 & 3)) add(slot(2), on(slot(2), 3, nprod) - (int)(rn >> 4 & 3));
        if ((pn & 3) && !on(slot(3), 0, nreac)) add(slot(3), (int)(pn & 3));
        if (nprod > 1 && (pn >> 2 & 3) && !on(slot(4), 0, nreac)) add(slot(4), (int)(pn >> 2 & 3));
        if (nprod > 2 && (pn >> 4 & 3) && !on(slot(5), 0, nreac)) add(slot(5), (int)(pn >> 4 & 3));
      } else {
        add(slot(0), -(int)(rn & 3));
        if (nreac > 1) add(slot(1), -(int)(rn >> 2 & 3));
        if (nreac > 2) add(slot(2), -(int)(rn >> 4 & 3));
        add(slot(3), (int)(pn & 3));
        if (nprod > 1) add(slot(4), (int)(pn >> 2 & 3));
        if (nprod > 2) add(slot(5), (int)(pn >> 4 & 3));
      }
    } else {
      wd[slot(0)] -= q;
      if (nreac > 1) wd[slot(1)] -= q;
      if (nreac > 2) wd[slot(2)] -= q;
      wd[slot(3)] += q;
      if (nprod > 1) wd[slot(4)] += q;
      if (nprod > 2) wd[slot(5)] += q;
    }
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
// TEAM: every sum in the order of team_rhs, whose values it then returns bit for
// bit (ck_rhs, where the batch chooses between the two; at most 64 species).
// Otherwise one species and one slot after another (RKF45, whose last reactors
// teams take over in that order).
template <bool INT, bool TEAM, bool WHOLE>
__device__ __forceinline__ void rhs_thread(const MechView& m, double p, const double* y, int ys,
                                           double* f, int fs, double* X, double* G, double* wd) {
  const int S = m.S;
  const double T = y[0];
  const double invT = __drcp_rn(T);
  const double lnT = log(T);
  const double log2T = lnT * INV_LN2;
  const double T2 = T * T, T3 = T2 * T, T4 = T3 * T;
  auto moles = [&](int k) { return __dmul_rn(y[(1 + k) * ys], m.invW[k]); };
  double sumYW = 0.0;
  if constexpr (TEAM) sumYW = tree_sum<double>(S, moles);
  else
    for (int k = 0; k < S; ++k) sumYW = fma(y[(1 + k) * ys], m.invW[k], sumYW);
  const double rho = m.cv ? p : p / (R_GAS * T * sumYW);
  bool in = INT && temp_in_range(T);
  double Ctot = 0.0;
  for (int k = 0; k < S; ++k) {
    const double xk = __dmul_rn(rho, moles(k));
    X[k] = xk;
    if (!TEAM) Ctot += xk;
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
  if constexpr (TEAM) Ctot = tree_sum<double>(S, [&](int k) { return X[k]; });
  const double* Gm = G + S;
  if constexpr (INT) {
    if (__all_sync(__activemask(), in)) rates_thread<true, TEAM, WHOLE>(m, T, invT, log2T, Ctot, X, G, Gm, wd);
    else rates_thread<false, TEAM, WHOLE>(m, T, invT, log2T, Ctot, X, G, Gm, wd);
  } else {
    rates_thread<false, TEAM, WHOLE>(m, T, invT, log2T, Ctot, X, G, Gm, wd);
  }
  const double invrho = __drcp_rn(rho);
  const double cvf = m.cv ? 1.0 : 0.0;
  double cpm = 0.0, hw = 0.0;
  for (int k = 0; k < S; ++k) {
    const double* a = m.th + k * TH_PER_SPECIES + (T < m.tmid[k] ? 0 : TH_STRIDE);
    double cp = fma(a[4], T4, fma(a[3], T3, fma(a[2], T2, fma(a[1], T, a[0])))) - cvf;
    double h = fma(a[10], invT, fma(a[9], T4, fma(a[8], T3, fma(a[7], T2, fma(a[6], T, a[5]))))) - cvf;
    const double w = wd[k];
    if constexpr (TEAM) {  // the terms, in the Gibbs factors' place
      G[k] = fma(moles(k), cp, 0.0);
      G[S + k] = fma(h, w, 0.0);
    } else {
      cpm = fma(moles(k), cp, cpm);
      hw = fma(h, w, hw);
    }
    f[(1 + k) * fs] = w * (m.W[k] * invrho);
  }
  if constexpr (TEAM) {
    const Two sums = tree_sum<Two>(S, [&](int k) { return Two{G[k], G[S + k]}; });
    cpm = sums.a;
    hw = sums.b;
  }
  f[0] = -T * hw / (rho * cpm);
}

}  // namespace ck
