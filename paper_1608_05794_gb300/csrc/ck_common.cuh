// Device-side data layout and arithmetic shared by the CUDA kernels of the
// batched constant-pressure reactor library (Stone, Alferman & Niemeyer,
// arXiv 1608.05794, Sec. 3 source terms; Sec. 2 integrators).
//
// FP64 is the scarce resource on this GPU (about 1.2 TFLOP/s against
// 70 TFLOP/s FP32), so the tables are pre-scaled at load time to save FP64
// instructions at run time: rate constants are kept as base-2 logarithms
// and evaluated with a table-driven 2^x (8 FP64 instructions), and the
// Gibbs polynomials are pre-divided by ln 2.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace ck {

constexpr double R_GAS = 8.314462618;       // J/(mol K)
constexpr double P_STD = 101325.0;          // p0 of Eq. kc, Pa
constexpr double LN2 = 0.6931471805599453094;
constexpr double INV_LN2 = 1.4426950408889634074;
constexpr double R_OVER_P0 = R_GAS / P_STD;               // R T / p0 is the molar volume at p0, m^3/mol
constexpr double P0_OVER_R = P_STD / R_GAS;

// One reaction, 112 bytes, read uniformly by all lanes (thread-per-reactor
// kernels) or by one lane per reaction (team kernels, in 16-byte loads; the
// last two hold the fall-off limit and are loaded for fall-off reactions
// only).  The loader sorts the reactions by (type, reversible, reactant
// count, product count) so that neighbouring lanes of a team kernel take the
// same branches.
struct __align__(16) RxnRec {
  double lA2;    // log2 A (SI)
  double beta;   // temperature exponent
  double EoR2;   // Ea / (R ln 2), K
  double EoR;    // EoR2 * LN2 (as rounded by that product): d ln k_f/dT
  int16_t sp[6];    // reactant slots 0..2, product slots 3..5, padded with S
  int8_t type;      // 0 elementary, 1 third-body, 2 Lindemann
  int8_t rev;       // 1 reversible through K_c, 2 explicit reverse Arrhenius
  int8_t dnu;
  int8_t nreac;
  int8_t nprod;
  uint8_t repeats;  // species in more than one slot: REP_*
  int16_t eff_beg, eff_cnt;  // slice of the efficiency table (eff - 1 != 0)
  int16_t rev_ix;            // rev == 2: row of the explicit reverse table
  double dnu_d;    // sum of product minus reactant coefficients, as FP64
  double nreac_d;  // reactant count, as FP64
  double nprod_d;  // product count, as FP64
  double lA02;   // Lindemann low-pressure limit: log2 A0
  double beta0;
  double E0oR2;
  double E0oR;   // E0oR2 * LN2
};
static_assert(sizeof(RxnRec) == 112, "RxnRec layout");
// RxnRec::repeats: which slots of a side hold the same species (reactants in the
// low three bits, products in the next three), and whether a species is on both
// sides.  REP_NET has 2 bits a slot, 6 a pattern: how often the species of a slot
// is in the pattern's side, in its first slot, else 0.
enum : uint8_t { REP_NONE = 0, REP_01 = 1, REP_02 = 2, REP_12 = 3, REP_ALL = 4, REP_BOTH_SIDES = 64 };
constexpr uint32_t REP_NET = (1u | 1u << 2 | 1u << 4) | (2u | 1u << 4) << 6 | (2u | 1u << 2) << 12 |
                             (1u | 2u << 2) << 18 | 3u << 24;

// Per-reaction values of a chunk of c reactions that the Jacobian is
// assembled from: q, dq/dT and D (c each), six partials a reaction (reactant
// slots 0..2, product slots 3..5), and dc/d[M] (k_f prod' - k_r prod'') of
// the chunk's third-body and fall-off reactions (its last ones).
constexpr int JAC_PER_RXN = 9;

// Per species and temperature range: 18 doubles
//   cp/R  : c0 + c1 T + c2 T^2 + c3 T^3 + c4 T^4               [0..4]
//   H/RT  : h0 + h1 T + h2 T^2 + h3 T^3 + h4 T^4 + h5 / T       [5..10]
//   g/ln2 : (S/R - H/RT)/ln 2 = G0 ln T + G1 + G2 T + G3 T^2 + G4 T^3 + G5 T^4 + G6 / T   [11..17]
constexpr int TH_STRIDE = 18;
constexpr int TH_PER_SPECIES = 2 * TH_STRIDE;

// Packed team-kernel table records (one 16-byte load each).
struct __align__(16) CsrTerm {  // species -> reaction list: net coefficient and reaction
  double nu;
  int32_t rx, pad;
};
struct __align__(16) JcEntry {  // one species-block entry of the Jacobian assembly
  int32_t idx;                  // flat index of the target (see JacTab)
  int32_t beg, end;             // its contribution terms
  int32_t pad;
};
struct __align__(16) JcTerm {   // coef * P[pidx]
  double coef;
  int32_t pidx, pad;
};
static_assert(sizeof(CsrTerm) == 16 && sizeof(JcEntry) == 16 && sizeof(JcTerm) == 16, "packed records");

// One way of assembling the Jacobian: the reactions in chunks of `chunk`
// (scratch doubles of per-reaction values), and per chunk c the targets
// jc[e], e in [jc_ptr[c], jc_ptr[c+1]) (flat index idx: the species-block
// entry J[idx], rows ld apart, below n ld, else the per-species sums wd, aT,
// E, u at idx - n ld), which add the sum over t in [jc[e].beg, jc[e].end) of jt[t].coef *
// src[jt[t].pidx] (src: the chunk's per-reaction values).  Chunk 0 lists
// every target, those without a term too.
struct JacTab {
  int chunk, n_chunks, scratch, ld;
  const int32_t* jc_ptr;
  const JcEntry* jc;
  const JcTerm* jt;
};

// Device view of a loaded mechanism.  All pointers are device memory (one
// allocation, 16-byte aligned sections).
struct DevMech {
  int S, R, n;            // species, reactions, n = S + 1
  int n_eff;              // entries of the efficiency table
  int csr_nnz;            // entries of the species -> reaction table
  int all_same_tmid;      // every species shares one T_mid
  int cv;                 // 1: constant volume (the parameter is rho), 0: constant pressure
  double tmid0;
  const RxnRec* rxn;      // [R]
  const double* thermo;   // [S][2][TH_STRIDE]
  const double* tmid;     // [S]
  const double* W;        // [S] kg/mol
  const double* invW;     // [S]
  const int16_t* eff_sp;  // [n_eff]
  const double* eff_m1;   // [n_eff] efficiency - 1
  const int32_t* csr_ptr; // [S+1] species -> (reaction, net nu) lists
  const CsrTerm* csr;     // [csr_nnz]
  const int32_t* slot_ptr;  // [S+1] species -> its reaction slots one by one, -1 a reactant, +1 a product,
  const CsrTerm* slot;      // in the order in which RKF45's threads add them (at most 32 species)
  const double* tab;      // [256] 2^(j/256)
  const double* revp;     // [n_rev][3] explicit reverse: log2 A_r, beta_r, Ea_r / (R ln 2)
  // A right-hand side whose team has no room for all R rates takes the
  // reactions in chunks of rhs_chunk.  csr_cptr[k (n_rhs_chunks + 1) + c] =
  // first CSR entry of species k whose reaction lies in chunk c or later.
  int rhs_chunk, n_rhs_chunks;
  int first_typed;        // reactions from here on are third-body or fall-off
  const int32_t* csr_cptr;
  // Jacobian tables: for teams that may assemble in device memory (the
  // per-reaction values then take the place of the matrix in shared memory,
  // usually of all reactions at once), and for those that may not.
  JacTab wide, narrow;
  const int16_t* rsp;     // [S] species order of the RHS gather, longest row first
};

// ---------------------------------------------------------------- 2^x
// Table-driven 2^x after Tang, "Table-driven implementation of the
// exponential function in IEEE floating-point arithmetic" (ACM TOMS 15,
// 1989), in base 2: x = e + j/256 + r with |r| <= 1/512, 2^x = 2^e T_j 2^r,
// T_j = 2^(j/256) from a 256-entry table, 2^r - 1 by its degree-4 Taylor
// polynomial in r ln 2 (truncation < 4e-17 relative).  The reduction is
// exact (x - round_{1/256}(x) is representable), so the result is within
// about one ulp.  |x| > 1000 (and NaN) falls back to the library exp2, out of
// line so that the rarely taken branch adds no instructions to the inlined
// fast path.  The range test compares the bits of |x| as an integer (they
// order like |x|, NaN above +inf), which keeps it off the FP64 pipe.
static __device__ __noinline__ double ck_exp2_wide(double x) { return exp2(x); }

__device__ __forceinline__ bool ck_exp2_in_range(double x) {
  const unsigned long long ax = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffULL;
  return ax <= 0x408F400000000000ULL;  // the bits of 1000.0
}

// 2^r - 1 for |r| <= 1/512 (Taylor, degree 4 in r ln 2), and the step that
// assembles 2^(e + j/256 + r) from it.
__device__ __forceinline__ double ck_exp2_poly(double r) {
  const double c1 = 0.69314718055994530942;
  const double c2 = 0.24022650695910071233;   // ln2^2/2
  const double c3 = 0.055504108664821579953;  // ln2^3/6
  const double c4 = 0.0096181291076284771620; // ln2^4/24
  return fma(fma(fma(c4, r, c3), r, c2), r, c1) * r;
}
__device__ __forceinline__ double ck_exp2_assemble(int i, double q, const double* __restrict__ tab) {
  const int j = i & 255;
  const int e = i >> 8;  // floor division by 256
  const double tj = tab[j];
  const double res = fma(tj, q, tj);
  return __longlong_as_double(__double_as_longlong(res) + ((long long)e << 52));
}

__device__ __forceinline__ double ck_exp2(double x, const double* __restrict__ tab) {
  if (!ck_exp2_in_range(x)) return ck_exp2_wide(x);
  const double SHIFT = 26388279066624.0;  // 1.5 * 2^44: ulp 2^-8
  const double t = x + SHIFT;
  const double r = x - (t - SHIFT);
  const int i = (int)__double2loint(t);  // round(x * 256), low bits of t
  return ck_exp2_assemble(i, ck_exp2_poly(r), tab);
}

// 2^x and 2^-x from one reduction.  Rounding x to a multiple of 1/256 is
// symmetric (ties to even), so -x reduces to -i and -r exactly, and both
// results are bitwise those of ck_exp2(x) and ck_exp2(-x).
__device__ __forceinline__ void ck_exp2_pm(double x, const double* __restrict__ tab, double& ep, double& em) {
  if (!ck_exp2_in_range(x)) {
    ep = ck_exp2_wide(x);
    em = ck_exp2_wide(-x);
    return;
  }
  const double SHIFT = 26388279066624.0;
  const double t = x + SHIFT;
  const double r = x - (t - SHIFT);
  const int i = (int)__double2loint(t);
  ep = ck_exp2_assemble(i, ck_exp2_poly(r), tab);
  em = ck_exp2_assemble(-i, ck_exp2_poly(-r), tab);
}

// 1 / x rounded to nearest: the value IEEE division 1 / x returns, without
// the general-division path.
__device__ __forceinline__ double rcp_rn(double x) { return __drcp_rn(x); }
__device__ __forceinline__ float rcp_rn(float x) { return __frcp_rn(x); }

// (R T / p0)^dnu for dnu = nprod - nreac in [-2, 2]: the concentration
// factor of 1/K_c (Eq. kc), by multiplication instead of an exponential.
__device__ __forceinline__ double rt_over_p0_pow(int dnu, double T, double invT) {
  const double q = dnu >= 0 ? T * R_OVER_P0 : invT * P0_OVER_R;
  const int a = dnu >= 0 ? dnu : -dnu;
  return a == 0 ? 1.0 : (a == 1 ? q : q * q);
}

// ---------------------------------------------------------------- products off the FP64 pipe
// a * b rounded to nearest even, in integer arithmetic: the 53-bit
// significands are multiplied in full (b's shifted up by 11, so that the upper
// 64 bits of the product hold the result and the lower 64 its rounding), the
// leading bit normalised and the rest rounded.  About 42 issue cycles of one
// scheduler; the FP64 unit, which the SM's four schedulers share, takes 64 of
// them for a warp instruction, and the integer units are idle beside it.  The
// same bits as the FP64 instruction while both operands and the product are
// normal numbers (nothing else is handled: callers check the ranges).
__device__ __forceinline__ double mul_int(double a, double b) {
  const uint32_t ah = (uint32_t)__double2hiint(a), al = (uint32_t)__double2loint(a);
  const uint32_t bh = (uint32_t)__double2hiint(b), bl = (uint32_t)__double2loint(b);
  const uint32_t mh = (ah & 0xfffffu) | 0x100000u, nh = (bh & 0xfffffu) | 0x100000u;
  const uint32_t Bh = __funnelshift_l(bl, nh, 11), Bl = bl << 11;
  const uint64_t t0 = (uint64_t)al * Bl;
  const uint64_t t1 = (uint64_t)al * Bh + (uint32_t)(t0 >> 32);
  const uint64_t t2 = (uint64_t)mh * Bl + (uint32_t)t1;
  const uint64_t t3 = (uint64_t)mh * Bh + (uint32_t)(t1 >> 32) + (uint32_t)(t2 >> 32);
  uint32_t H1 = (uint32_t)(t3 >> 32), H0 = (uint32_t)t3, L1 = (uint32_t)t2;
  const uint32_t L0 = (uint32_t)t0;
  const int s = (int)(H1 >> 20) ^ 1;  // 1: the product of the significands is below 2
  H1 = __funnelshift_l(H0, H1, s);
  H0 = __funnelshift_l(L1, H0, s);
  L1 = __funnelshift_l(L0, L1, s);
  const uint32_t sticky = (L1 << 1) | L0;
  const uint32_t up = (L1 >> 31) & (H0 | (sticky != 0 ? 1u : 0u));
  const uint64_t m = (((uint64_t)H1 << 32) | H0) + (up & 1u);
  // biased exponents add up; the leading bit of m adds the last one
  const int e = (int)((ah >> 20) & 0x7ff) + (int)((bh >> 20) & 0x7ff) - 1023 - s;
  const uint32_t rh = ((uint32_t)e << 20) + (uint32_t)(m >> 32);
  return __hiloint2double((int)(rh | ((ah ^ bh) & 0x80000000u)), (int)(uint32_t)m);
}
// 1 / x rounded to nearest (the value IEEE division 1 / x returns), in integer
// arithmetic, off the FP64 unit: with M the 53-bit significand, 2^105 / M by
// Newton's iteration (z <- z + z (1 - z m)) from an FP32 estimate, the
// truncated quotient made exact by its remainder, which then rounds it (a tie
// is impossible: M does not divide an odd multiple of a power of two).  Errors:
// w 2^-29, q less than 2 units, so one correction each way is enough.  Powers
// of two and the ends of the exponent range take the library's reciprocal.
// Latency 284 cycles against 354 of __drcp_rn, whose seven FP64 instructions
// hold the shared unit for 112.
__device__ __forceinline__ double rcp_int(double x) {
  const uint32_t xh = (uint32_t)__double2hiint(x), xl = (uint32_t)__double2loint(x);
  const uint32_t ef = (xh >> 20) & 0x7ff;
  if (ef - 2u >= 2040u || (xl | (xh & 0xfffffu)) == 0) return __drcp_rn(x);
  const uint32_t mh = (xh & 0xfffffu) | 0x100000u;
  const uint64_t M = ((uint64_t)mh << 32) | xl;  // m = M / 2^52 in (1, 2)
  const uint32_t top = __funnelshift_l(xl, mh, 11);  // M >> 21
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(0x3f800000u | ((top >> 8) & 0x7fffffu))));
  const uint32_t v = (uint32_t)(y * 1073741824.0f);                     // 2^30 / m
  const int64_t e1 = (int64_t)((1ull << 61) - (uint64_t)v * top);      // 2^61 (1 - v m / 2^30)
  const uint32_t w = (v << 1) + (uint32_t)(int32_t)(((int64_t)(int32_t)v * (int32_t)(e1 >> 10)) >> 50);  // 2^31 / m
  // 2^83 (1 - w m / 2^31), below 2^54 in magnitude: its low 64 bits suffice
  const int64_t e2 = (int64_t)(0 - ((uint64_t)w * xl + ((uint64_t)(w * mh) << 32)));
  uint64_t q = ((uint64_t)w << 22) + (uint64_t)(((int64_t)(int32_t)(e2 >> 24) * (int64_t)(uint64_t)w) >> 37);
  int64_t rem = (int64_t)(0 - q * M);  // 2^105 - q M likewise
  if (rem < 0) {
    --q;
    rem += (int64_t)M;
  }
  if (rem >= (int64_t)M) {
    ++q;
    rem -= (int64_t)M;
  }
  q += (uint64_t)(2 * rem > (int64_t)M);
  // q in [2^52, 2^53): its leading bit adds the last one to the exponent field
  const uint32_t rh = (xh & 0x80000000u) | (((2044u - ef) << 20) + (uint32_t)(q >> 32));
  return __hiloint2double((int)rh, (int)(uint32_t)q);
}
__device__ __forceinline__ float rcp_int(float x) { return __frcp_rn(x); }
template <bool INT>
__device__ __forceinline__ double rcp_sel(double x) {
  if constexpr (INT) return rcp_int(x);
  else return __drcp_rn(x);
}
template <bool INT>
__device__ __forceinline__ double mul_sel(double a, double b) {
  if constexpr (INT) return mul_int(a, b);
  else return __dmul_rn(a, b);
}

// Ranges in which the products of a reaction's concentrations and Gibbs
// factors stay normal: up to three concentrations within 2^+-300 (not zero),
// and (R T/p0)^dnu, within 2^+-46 for T in [2^-9, 2^21), times up to six
// factors 2^(+-g), |g| < 160.
__device__ __forceinline__ bool conc_in_range(double x) {
  const uint32_t e = ((uint32_t)__double2hiint(x) >> 20) & 0x7ff;
  return e - (1023u - 300u) < 600u;
}
__device__ __forceinline__ bool gibbs_in_range(double g) {
  return ((uint32_t)__double2hiint(g) & 0x7fffffffu) < 0x40640000u;  // |g| < 160
}
__device__ __forceinline__ bool temp_in_range(double T) {
  const uint32_t h = (uint32_t)__double2hiint(T);
  return h - 0x3f600000u < 0x41400000u - 0x3f600000u;
}
// c k_f and c k_r within 2^+-400: their products with two concentrations are
// normal too.
__device__ __forceinline__ bool rate_in_range(double k) {
  const uint32_t e = ((uint32_t)__double2hiint(k) >> 20) & 0x7ff;
  return e - (1023u - 400u) < 800u;
}

// ---------------------------------------------------------------- statuses
enum : int32_t { ST_OK = 0, ST_MAXSTEPS = 1, ST_HMIN = 2, ST_NONFINITE = 3, ST_SINGULAR = 4,
                 ST_BADINPUT = 5 };

// Step-control constants (the paper leaves the controller unspecified; these
// are the readings shared with the CPU oracle's documentation).
constexpr double FAC_MAX = 5.0, FAC_MIN = 0.2, SAFETY = 0.9;
constexpr int SINGULAR_LIMIT = 10;

// ROS4 coefficients, App. C Table ros4 (gamma is the table value 0.57282;
// the table's b_i are the transformed-scheme weights m_i; a4j = a3j, a43 = 0
// so the fourth stage reuses the third stage's f).
constexpr double ROS_GAMMA = 0.57282;
constexpr double ROS_A21 = 2.0;
constexpr double ROS_A31 = 1.867943637803922, ROS_A32 = 0.2344449711399156;
constexpr double ROS_C21 = -7.137615036412310;
constexpr double ROS_C31 = 2.580708087951457, ROS_C32 = 0.6515950076447975;
constexpr double ROS_C41 = -2.137148994382534, ROS_C42 = -0.3214669691237626,
                 ROS_C43 = -0.6949742501781779;
constexpr double ROS_M1 = 2.255570073418735, ROS_M2 = 0.2870493262186792,
                 ROS_M3 = 0.4353179431840180, ROS_M4 = 1.093502252409163;
constexpr double ROS_E1 = -0.2815431932141155, ROS_E2 = -0.07276199124938920,
                 ROS_E3 = -0.1082196201495311, ROS_E4 = -1.093502252409163;

// RKF45 tableau, App. B Table rkf45 (b: fourth-order weights, propagated;
// bh: fifth-order weights; the error is sum (bh - b) k).
constexpr double RK_A21 = 1.0 / 4.0;
constexpr double RK_A31 = 3.0 / 32.0, RK_A32 = 9.0 / 32.0;
constexpr double RK_A41 = 1932.0 / 2197.0, RK_A42 = -7200.0 / 2197.0, RK_A43 = 7296.0 / 2197.0;
constexpr double RK_A51 = 439.0 / 216.0, RK_A52 = -8.0, RK_A53 = 3680.0 / 513.0,
                 RK_A54 = -845.0 / 4104.0;
constexpr double RK_A61 = -8.0 / 27.0, RK_A62 = 2.0, RK_A63 = -3544.0 / 2565.0,
                 RK_A64 = 1859.0 / 4104.0, RK_A65 = -11.0 / 40.0;
constexpr double RK_B1 = 25.0 / 216.0, RK_B3 = 1408.0 / 2565.0, RK_B4 = 2197.0 / 4104.0,
                 RK_B5 = -1.0 / 5.0;
constexpr double RK_D1 = 16.0 / 135.0 - 25.0 / 216.0, RK_D3 = 6656.0 / 12825.0 - 1408.0 / 2565.0,
                 RK_D4 = 28561.0 / 56430.0 - 2197.0 / 4104.0, RK_D5 = -9.0 / 50.0 + 1.0 / 5.0,
                 RK_D6 = 2.0 / 55.0;

// Per-CTA global scratch of the ROS4 kernel, in doubles: -J of the current
// state (n x n) and its diagonal (n).
__host__ __device__ constexpr size_t ros4_scratch_doubles(int n) { return (size_t)n * n + (size_t)n; }

// A reactor that the thread-per-reactor RKF45 hands to a team part-way (its
// state is in the caller's y).
struct RkCont {
  double t, h;
  int32_t r, acc, rej;
  int16_t last_rej, last_nf;
};

struct SolverParams {
  double rtol, atol, h0, fixed_h;
  int max_steps;
  int jac;  // ROS4 Jacobian: 0 analytic, 1 forward differences
};

}  // namespace ck
