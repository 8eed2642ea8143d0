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

// Room for a right-hand side's rates of progress (team_rhs, team_rhs_lat).
// The latency form, which takes all reactions at once, keeps one more value of
// each third-body and fall-off reaction.
__host__ __device__ __forceinline__ int rhs_doubles(const DevMech& d) {
  return d.rhs_chunk + (d.S <= 32 && d.R <= d.rhs_chunk ? d.R - d.first_typed : 0);
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

// Most reactions of a chunk of the right-hand side, of the wide and of the
// narrow Jacobian (all of them at once where they fit).
struct TeamChunks {
  int rhs, wide, narrow;
};
__host__ inline TeamChunks team_chunks(int S, int R, int typed) {
  const int n = S + 1;
  auto shares = [&](int most) { return R ? (R + (R + most - 1) / most - 1) / ((R + most - 1) / most) : 1; };
  // the wide form's scratch takes the matrix's place in shared memory: all
  // reactions at once where they fit it (or 24 KB)
  const int room = n * n > 3072 ? n * n : 3072;
  TeamChunks c;
  c.rhs = shares(n <= 64 ? 512 : 392);
  c.wide = JAC_PER_RXN * R + typed <= room ? (R > 1 ? R : 1) : shares(room / (JAC_PER_RXN + 1));
  c.narrow = shares(n <= 64 ? 64 : 60);
  return c;
}

}  // namespace ck
