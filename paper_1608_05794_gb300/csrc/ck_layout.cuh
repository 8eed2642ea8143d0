// Shared-memory layout of the team kernels: sizes in doubles, the same on the
// host (launch sizes) and on the device (offsets).
#pragma once
#include "ck_common.cuh"

namespace ck {

// Species arrays of a team (TeamBufs) up to wd; a Jacobian continues with
// three of S.
constexpr int TEAM_RED_DOUBLES = 64;
__host__ __device__ __forceinline__ constexpr int species_doubles(int S) { return TEAM_RED_DOUBLES + 4 * (S + 1) + 2 * S; }

// Distance of the rows of a factored matrix in shared memory: odd, so that
// the lanes of a warp reading one column (a row each: the pivot search, the
// substitutions) touch different banks.  At n = 112 every such load took 32
// turns.
__host__ __device__ __forceinline__ constexpr int lu_ld(int n) { return n | 1; }

// Dynamic shared memory, in doubles, with which `ctas` of them fit an SM: 228 KB
// an SM and 227 KB a CTA, less the 1 KB that every CTA reserves and 80 bytes of
// static shared memory (k_ros4's step control).
__host__ __device__ __forceinline__ constexpr int smem_doubles(int ctas) {
  return ((ctas > 1 ? 228 * 1024 / ctas - 1024 : 227 * 1024) - 80) / 8;
}

// Where a right-hand side keeps its rates of progress: offset in shared
// memory and how many at a time (all m.R, or m.rhs_chunk).
struct RhsQ {
  int off, chunk;
};

// Mechanisms that the latency kernels take in the latency form: at most 32
// species and 64 reactions, of which one warp forms the rate constants in two
// rounds.  With more its chain is the longer one: RKF45 on 500 reactors of 10
// species, latency form / general, ms: 20 reactions 6.7 / 8.9, 60 8.5 / 10.1,
// 100 12.7 / 11.5, 280 22.0 / 19.4, 600 41.1 / 31.3; 30 species: 60 reactions 3.9 /
// 5.0, 120 6.0 / 5.5.
constexpr int LAT_REACTIONS = 64;
__host__ __device__ __forceinline__ bool latency_form(const DevMech& d) { return d.S <= 32 && d.R <= LAT_REACTIONS; }

// Room for a right-hand side's rates of progress (team_rhs, team_rhs_lat).
// The latency form keeps one more value of each third-body and fall-off
// reaction.
__host__ __device__ __forceinline__ int rhs_doubles(const DevMech& d) {
  return d.rhs_chunk + (latency_form(d) ? d.R - d.first_typed : 0);
}

// Shared memory of one k_ros4 CTA, in doubles: the matrix, y and f(y), the team's work arrays, and the stage vectors,
// the factors' row table and the rates of progress (or the LU's scratch).  The
// Jacobian's per-reaction values lie over the matrix (wide: it is assembled in
// device memory) or behind the work arrays, over the stage vectors.
struct Ros4Layout {
  int vp, yv, f0, bufs, jscr, yt, ub, invd, rof, lr;
  RhsQ rhs_q;
  size_t doubles;
  __host__ __device__ Ros4Layout(const DevMech& d, bool wide) {
    const int n = d.n, mat = n * lu_ld(n);
    vp = n > 64 ? 256 : 64;
    yv = wide && d.wide.scratch > mat ? d.wide.scratch : mat;
    f0 = yv + n;
    bufs = f0 + n;
    const int t = bufs + species_doubles(d.S), tj = t + 3 * d.S;
    jscr = wide ? 0 : tj;
    yt = t;
    ub = yt + n;
    invd = ub + n;
    rof = invd + n;
    const int after = (rof + (n + 1) / 2 + 1) & ~1;  // 16-byte aligned
    lr = after;
    rhs_q.off = after;
    rhs_q.chunk = d.rhs_chunk;
    int most = wide ? tj : tj + d.narrow.scratch;
    if (after + 4 * n > most) most = after + 4 * n;
    if (after + rhs_doubles(d) > most) most = after + rhs_doubles(d);
    doubles = (size_t)most;
  }
};

// CTAs an SM that shared memory is shared out for: what the registers of the
// kernels with a matrix allow (launch bounds), for n <= 24 fewer, where a larger
// share holds more of a mechanism of many reactions (10 species, 280 reactions,
// ROS4 on 500 reactors: 31.9 ms with eight, 33.0 with twelve).
__host__ __device__ __forceinline__ constexpr int team_ctas(int n) { return n <= 24 ? 8 : (n <= 64 ? 6 : 2); }

// Reactions at a time of the right-hand side, of the wide and of the narrow
// Jacobian of k_ros4: all of them where they fit the shared memory that the
// residency leaves, else equal shares.
struct TeamChunks {
  int rhs, wide, narrow;
};
__host__ inline TeamChunks team_chunks(int S, int R, int typed) {
  const int n = S + 1, mat = n * lu_ld(n);
  // Ros4Layout up to the rates
  const int before = (mat + 5 * n + (n + 1) / 2 + 1 + species_doubles(S)) & ~1;
  int ctas = team_ctas(n);
  while (ctas > 1 && smem_doubles(ctas) < before + 4 * n) --ctas;
  auto shares = [&](int most) { return (R + (R + most - 1) / most - 1) / ((R + most - 1) / most); };
  TeamChunks c{1, 1, 1};
  if (R == 0) return c;
  // (that of the latency form, at most 128 of the rates, is always there)
  const int rates = smem_doubles(ctas) - before, factors = S <= 32 && R <= LAT_REACTIONS ? typed : 0;
  c.rhs = R <= rates ? R : shares(rates);
  const int beside = c.rhs + factors;
  // the wide form's values lie over the matrix, the narrow one's behind the work
  // arrays
  int over = mat + rates - (beside > 4 * n ? beside : 4 * n);
  // (and leave k_jacobian, which has no matrix, the same residency)
  const int alone = smem_doubles(team_ctas(n)) - (2 * n + species_doubles(S) + 3 * S);
  if (alone < over) over = alone;
  c.wide = JAC_PER_RXN * R + typed <= over ? R : shares(over / (JAC_PER_RXN + 1));
  const int behind = smem_doubles(ctas) - (mat + 2 * n + species_doubles(S) + 3 * S);
  c.narrow = JAC_PER_RXN * R + typed <= behind ? R : shares(behind / (JAC_PER_RXN + 1));
  return c;
}

}  // namespace ck
