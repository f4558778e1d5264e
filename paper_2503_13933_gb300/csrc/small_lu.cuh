// LU with partial pivoting of one M x M system (M <= TAPS_MAX_M) in shared memory by one CTA,
// the right-hand side carried along as column M.
//
// A step's pivot work is a chain of its own (search, reciprocal, multipliers: ~1200 clocks)
// beside the trailing update's FP64 issue ((M - p)^2 / 2 clocks), so the two overlap: during
// step p warp 0 updates column p + 1 first, finds its pivot row (largest magnitude, ties to
// the smaller row; integer compares of the magnitudes' bit patterns), takes the reciprocal
// (seed plus refinement) and forms the next step's multipliers l_r = T[r][p+1] / pivot with the
// lanes over the rows, while warps 1 .. update the other columns, one FMA per entry,
// T[r][c] -= l_r T[p][c], the threads dealt out over the whole trailing block so that no lane
// idles at row ends.  Rows change places in a table of row offsets, not in memory, and a step
// has one barrier.  Warp 0 then substitutes back alone, its lanes holding the right-hand side,
// with the kept reciprocals (0 for a zero or non-finite pivot, which sets `bad`).  Every entry
// takes the same FMAs in the same order as with two barriers per step and the pivot search
// between them.
#pragma once

#include "taps_internal.cuh"

struct SmallLu {   // in shared memory
  double invd[TAPS_MAX_M];      // reciprocals of the pivots
  double lmul[2][TAPS_MAX_M];   // multipliers of two steps, by row
  int rowat[2][TAPS_MAX_M];     // offset of row r in T, for two steps (rows from the step's on)
  int rowfin[TAPS_MAX_M];       // offsets of the pivot rows
};

// T: [M][M + 1], complete (the caller has synchronised); called by all NT threads.  On return
// lane l of warp 0 holds entries l, l + 32, ... of the solution in b.
template <int NT>
__device__ __forceinline__ void small_lu_solve(double* T, int M, SmallLu& sh, double (&b)[TAPS_MAX_M / 32], bool& bad) {
  constexpr int S = TAPS_MAX_M / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int ld = M + 1;
  for (int r = tid; r < M; r += NT) sh.rowat[0][r] = r * ld;
  __syncthreads();
  bad = false;
  // warp 0: the pivot of step p, whose column is final in T; rows in `at` order on entry,
  // `to` receives the step's order and `l` its multipliers
  auto pivot = [&](int p, const int* at, int* to, double* l) {
    double v[S];
    long long best = -1;
    int br = p;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const int r = p + lane + 32 * s;
      if (r < M) {
        v[s] = T[at[r] + p];
        const long long a = __double_as_longlong(fabs(v[s]));
        if (a > best) { best = a; br = r; }
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
      const long long ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int orr = __shfl_xor_sync(0xffffffffu, br, o);
      if (ob > best || (ob == best && orr < br)) { best = ob; br = orr; }
    }
    const double pv = T[at[br] + p];
    const bool ok = taps_finite_nonzero(pv);
    const double inv = ok ? taps_rcp(pv) : 0.0;
    bad |= !ok;
    if (lane == 0) {
      sh.invd[p] = inv;
      sh.rowfin[p] = at[br];
    }
    const double v0 = T[at[p] + p];   // the row that takes br's place
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const int r = p + lane + 32 * s;
      if (r < M) {
        to[r] = at[r == p ? br : (r == br ? p : r)];
        if (r > p) l[r] = (r == br ? v0 : v[s]) * inv;
      }
    }
  };
  if (warp == 0) pivot(0, sh.rowat[0], sh.rowat[1], sh.lmul[0]);
  __syncthreads();
  for (int p = 0; p < M; ++p) {
    const int* at = sh.rowat[(p + 1) & 1];   // the order of step p
    const double* l = sh.lmul[p & 1];
    const double* prow = T + sh.rowfin[p];
    if (warp == 0) {
      if (p + 1 < M) {
        const double pc = prow[p + 1];
        for (int r = p + 1 + lane; r < M; r += 32) {
          double* x = T + at[r] + p + 1;
          *x = fma(-l[r], pc, *x);
        }
        __syncwarp();
        pivot(p + 1, at, sh.rowat[p & 1], sh.lmul[(p + 1) & 1]);
      }
    } else {
      // columns p + 2 .. M of the rows after p, over warps 1 ..
      const int w = M - 1 - p, rows = M - 1 - p;   // (the right-hand side among the columns)
      if (w > 0) {
        const int t = tid - 32, nt = NT - 32;
        int r = t / w, c = t - r * w;
        const int dr = nt / w, dc = nt - dr * w;
        while (r < rows) {
          double* x = T + at[p + 1 + r] + p + 2 + c;
          *x = fma(-l[p + 1 + r], prow[p + 2 + c], *x);
          r += dr;
          c += dc;
          if (c >= w) {
            c -= w;
            ++r;
          }
        }
      }
    }
    __syncthreads();
  }
  if (warp != 0) return;
  // x_r in the lane that holds row r
  const int* at = sh.rowfin;
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const int r = lane + 32 * s;
    b[s] = r < M ? T[at[r] + M] : 0.0;
  }
#pragma unroll
  for (int sr = S - 1; sr >= 0; --sr) {
    for (int r = min(M - 1, 32 * sr + 31); r >= 32 * sr; --r) {
      const double xr = __shfl_sync(0xffffffffu, b[sr], r & 31) * sh.invd[r];   // 0 for a bad pivot
      if (lane == (r & 31)) b[sr] = xr;
#pragma unroll
      for (int s = 0; s <= sr; ++s) {
        const int k = lane + 32 * s;
        if (k < r) b[s] = fma(-T[at[k] + r], xr, b[s]);
      }
    }
  }
}
