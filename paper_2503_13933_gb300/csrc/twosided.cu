// Block-banded elimination from both ends (Eqs. 36-40, 43) on thread-block clusters.
//
// The reduced matrix of a dim is a block band: n nodes, M x M blocks, hb blocks on
// either side of the diagonal.  Its elimination is a chain of n dependent block rows, and
// on this GPU the chain, not the FP64 work, is what a solve costs (64 nodes, 10 modes:
// 3.8 MFLOP, 3 us at the FP64 peak; the one-ended cooperative elimination, two grid
// barriers per row, takes 1150 us with its back substitution).  Here:
//   - the chain is halved: one cluster eliminates the nodes from the low end, another the
//     nodes from the high end, until hb nodes are left in the middle, to which both sides'
//     Schur updates are added; a third cluster solves the middle and substitutes back
//     towards both ends at once.  Any order of elimination without pivoting exists, the
//     symmetric part of every reduced matrix being positive definite.
//   - a row costs one hardware cluster barrier instead of two grid barriers through global
//     memory.  The active window (hb + 1 nodes) lives in the cluster's shared memory, its
//     scalar columns dealt out to the CTAs; per node k every CTA forms W = D^-1 A(k, .) for
//     its own columns (factoring the diagonal block redundantly: M dependent pivots either
//     way) and subtracts A(., k) W from them.  The columns
//     of node k + 1 are updated first and pushed to every CTA of the cluster (distributed
//     shared memory), so the barrier's wait overlaps the rest of the update.
//   - entries of the band that enter the window, and the W blocks of the back
//     substitution, travel by cp.async a node ahead of their use.
// The panel of a node (its M columns) is held three times, the window once: up to M = 37 at
// hb = 5 in 227 KB; beyond that the one-ended elimination is the route.
#include <string.h>

#include <algorithm>
#include <type_traits>

#include <cooperative_groups.h>

#include "taps_internal.cuh"

namespace cg = cooperative_groups;

#define TS_THREADS 256
#define TS_COLS 64    // most columns of [D | own columns] per CTA
#define TS_STAGES 4   // W blocks in flight during the back substitution (fewer if they do not fit)

__device__ __forceinline__ void ts_copy8(double* smem, const double* gmem) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(gmem));
}
__device__ __forceinline__ void ts_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void ts_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void ts_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void ts_cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Quotient and remainder by a divisor fixed for the launch: one high product instead of an
// integer division (e d < 2^32, so the rounded-up reciprocal gives the exact quotient).
struct TsDiv {
  unsigned d, inv;
  __device__ __forceinline__ explicit TsDiv(int dd) : d(dd), inv(dd > 1 ? 0xffffffffu / (unsigned)dd + 1u : 0u) {}
  __device__ __forceinline__ int div(int e) const { return d > 1 ? (int)__umulhi((unsigned)e, inv) : e; }
  __device__ __forceinline__ int mod(int e) const { return e - div(e) * (int)d; }
};

// Shared memory of one CTA, in doubles.
struct TsLayout {
  int rows;   // (hb + 1) M: rows of the window
  int cw;     // own columns of the window
  size_t pan, win, rhs, wbuf, col, total;
};
__host__ __device__ inline TsLayout ts_layout(int hb, int M, int nc) {
  TsLayout L;
  L.rows = (hb + 1) * M;
  L.cw = (L.rows + nc - 1) / nc;
  size_t off = 0;
  L.pan = off;                       // [3][M][rows]: panels (node k's columns), column-major
  off += 3 * (size_t)M * L.rows;
  L.win = off;                       // [cw][rows]: own columns, rows as a ring of nodes
  off += (size_t)L.cw * L.rows;
  L.rhs = off;                       // [rows]: the right-hand side (the last CTA's)
  off += L.rows;
  L.wbuf = off;                      // [cw + 1][M]: W of the own columns
  off += (size_t)(L.cw + 1) * M;
  L.col = off;                       // [2][64]: the multipliers of two pivots
  off += 128;
  L.total = off;
  return L;
}

struct TsArgs {
  double* blocks;   // [n][2 hb + 1][M][M] the reduced band; W replaces A(k, k +- j)
  double* F;        // [n][M] right-hand side; z = D^-1 F replaces it
  double* mid;      // [2][hb M + 1][hb M] the middle as each side leaves it, column-major
  int n, hb, M;
  int nlo, nhi;     // nodes eliminated from the low and from the high end
  int nmid;         // nodes between them
  double* X;        // factor [M][n]
  double* Save;     // the factor before the solve
  int* status;
};

// W = D^-1 A(k, .) for the own columns of the window by LU without pivoting on [D | own
// columns] (no inverse is formed: D^-1 A as a product would lose another factor cond(D); and the
// rows above a pivot wait for the back substitution: eliminated at once, Gauss-Jordan, they
// leave residuals that grow with cond(D), 8e-14 where these are 2e-17 on a 24-mode block of
// condition 2e15).  Every entry takes the operations of the one-ended elimination in their
// order.  Four warps, one per SM sub-partition: an FP64 instruction holds its
// sub-partition's pipe ~64 clocks, and a second warp's would sit in the pivot chain (eight warps
// took 1240 clocks a pivot at M = 10).  Warp w holds the columns w, w + 4, ... with the rows on
// the lanes (S row slots).  Per step everyone reads the multipliers published by the pivot's
// owner; the owner of the next column updates that column first and publishes its multipliers
// (reciprocal by seed and refinement), the chain of the step, and its entries above the
// diagonal, final by then, for the back substitution.  After four pivots every warp's columns
// move down one register slot, so that the next pivot's column has a fixed place.  The back
// substitution needs no barrier: every warp takes its own columns through the published ones of
// U, with the kept reciprocals of its diagonal.  It is the price of the small residual: 64 nodes
// at s = 2 take 266 us a solve at M = 10 and 234 as Gauss-Jordan, 1372 and 1125 at M = 30.
// up[c * ld + r]: U above the diagonal, in the place of D, which is in registers by then.
// put(ci, row, w): the solution of own column ci (ncol of them).
__device__ __forceinline__ void ts_sync4(int id) { asm volatile("bar.sync %0, 128;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void ts_arrive4(int id) { asm volatile("bar.arrive %0, 128;" ::"r"(id) : "memory"); }

template <int S, typename Put>
__device__ __forceinline__ void ts_solve_node(double (&v)[TS_COLS / 4][S], int M, int ncol, double* colb, double* up,
                                              int ld, int* status, bool report, Put put) {
  constexpr int KC = TS_COLS / 4;
  const int lane = threadIdx.x & 31;
  const int w = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);   // the same in every lane: uniform branches
  const int tot = M + ncol;
  double rinv[S] = {};   // 1 / pivot of the lane's rows
  auto row_of = [&](const double (&x)[S], int p) {
    double rp = __shfl_sync(0xffffffffu, x[0], p & 31);
    if (S > 1) {
      const double r1 = __shfl_sync(0xffffffffu, x[S - 1], p & 31);
      if (p >> 5) rp = r1;
    }
    return rp;
  };
  // every row below p less its multiplier times row p
  auto update = [&](double (&x)[S], const double (&f)[S], int p) {
    const double rp = row_of(x, p);
#pragma unroll
    for (int s = 0; s < S; ++s) x[s] = fma(-f[s], rp, x[s]);
  };
  // the multipliers of pivot q, none above it; 1 / pivot in its row; U above it
  auto publish = [&](const double (&x)[S], int q) {
    const double piv = row_of(x, q);
    double inv = taps_rcp(piv);
    const bool ok = taps_finite_nonzero(piv);
    if (!ok) inv = 1.0;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const int r = lane + 32 * s;
      const double f = x[s] * inv;
      colb[(q & 1) * 64 + r] = r < q ? 0.0 : (r == q ? inv : f);
      if (r < q) up[q * ld + r] = x[s];
    }
    if (!ok && report && lane == 0) taps_flag(status, TAPS_DEV_SINGULAR);
  };
  // the columns of this warp from c0 (that of v[0]) on, less the multipliers f of pivot p;
  // v[0] is done with once the pivot has passed it.  Slots go in groups, so that their
  // shuffles are in flight together; slots past the last column hold zeros.
  auto others = [&](const double (&f)[S], int p, int c0, int passed) {
    if (c0 > passed) update(v[0], f, p);
    if (c0 + 4 < tot) {
      update(v[1], f, p);
      update(v[2], f, p);
      update(v[3], f, p);
    }
#pragma unroll
    for (int g = 4; g < KC; g += 4) {
      if (c0 + 4 * g >= tot) break;
#pragma unroll
      for (int k = g; k < g + 4; ++k) update(v[k], f, p);
    }
  };
  if (w == 0) publish(v[0], 0);
  ts_sync4(2);
  // pivot p; `next` holds column p + 1 in its owner.  The others wait for the owner's
  // multipliers, the owner for nobody: it arrives at the step's barrier once they are
  // published and updates its other columns after that (two barriers in turn keep its next
  // arrival apart).  Each lane reads back the rows it published itself.
  auto step = [&](int p, int c0, double (&next)[S]) {
    double f[S];
#pragma unroll
    for (int s = 0; s < S; ++s) {
      f[s] = colb[(p & 1) * 64 + lane + 32 * s];
      if (lane + 32 * s == p) {
        rinv[s] = f[s];
        f[s] = 0.0;
      }
    }
    const int q = p + 1;
    if (q < M && w == (q & 3)) {
      update(next, f, p);
      double keep[S];   // column q has had this update
#pragma unroll
      for (int s = 0; s < S; ++s) keep[s] = next[s];
      publish(next, q);
      __syncwarp();
      ts_arrive4(1 + (p & 1));
      others(f, p, c0, q);
#pragma unroll
      for (int s = 0; s < S; ++s) next[s] = keep[s];
    } else {
      others(f, p, c0, p);
      ts_sync4(1 + (p & 1));
    }
  };
  int c0 = w;
#pragma unroll 1
  for (int p = 0; p < M; p += 4) {
#pragma unroll 1
    for (int j = 0; j < 3 && p + j < M; ++j) step(p + j, c0, v[0]);
    if (p + 3 < M) {
      step(p + 3, c0, v[1]);
#pragma unroll
      for (int k = 0; k + 1 < KC; ++k)
#pragma unroll
        for (int s = 0; s < S; ++s) v[k][s] = v[k + 1][s];
      c0 += 4;
    }
  }
  // back substitution: the rows above r less U(., r) times row r, for the slots that hold own
  // columns (the first may hold one of D's), U's next column loaded ahead
  if (c0 < M) {
#pragma unroll
    for (int k = 0; k + 1 < KC; ++k)
#pragma unroll
      for (int s = 0; s < S; ++s) v[k][s] = v[k + 1][s];
    c0 += 4;
  }
  const int held = (tot - c0 + 3) >> 2;
  if (S == 1 && M <= 16) {
    // two columns to a slot, one to a half of the lanes: an FP64 instruction costs the same
    const int row = lane & 15, top = lane & 16;
    double x[KC / 2];
#pragma unroll
    for (int k = 0; k < KC / 2; ++k) {
      const double hi = __shfl_sync(0xffffffffu, v[2 * k + 1][0], row);
      x[k] = top ? hi : v[2 * k][0];
    }
    const double ri = __shfl_sync(0xffffffffu, rinv[0], row);
    auto back = [&](auto slots) {
      double u = row < M - 1 ? up[(M - 1) * ld + row] : 0.0;
#pragma unroll 1
      for (int r = M - 1; r >= 0; --r) {
        const double ur = u;
        u = row < r - 1 ? up[(r - 1) * ld + row] : 0.0;
#pragma unroll
        for (int k = 0; k < decltype(slots)::value; ++k) {
          const double xs = x[k] * ri, xr = __shfl_sync(0xffffffffu, xs, r + top);   // every lane
          const double y = fma(-ur, xr, x[k]);
          x[k] = row == r ? xs : y;
        }
      }
    };
    if (held > 4) back(std::integral_constant<int, KC / 2>{});
    else if (held > 2) back(std::integral_constant<int, 2>{});
    else if (held > 0) back(std::integral_constant<int, 1>{});
#pragma unroll
    for (int k = 0; k < KC / 2; ++k) {
      const int c = c0 + 8 * k + (top >> 2);
      if (row < M && c < tot) put(c - M, row, x[k]);
    }
    return;
  }
  auto back = [&](auto slots) {
    double u[S];
#pragma unroll
    for (int s = 0; s < S; ++s) u[s] = lane + 32 * s < M - 1 ? up[(M - 1) * ld + lane + 32 * s] : 0.0;
#pragma unroll 1
    for (int r = M - 1; r >= 0; --r) {
      double ur[S];
#pragma unroll
      for (int s = 0; s < S; ++s) {
        ur[s] = u[s];
        u[s] = lane + 32 * s < r - 1 ? up[(r - 1) * ld + lane + 32 * s] : 0.0;
      }
      // row r of slot k in lane k: one product with the reciprocal for all slots
      const double ir = row_of(rinv, r);
      double xp = 0.0;
#pragma unroll
      for (int k = 0; k < decltype(slots)::value; ++k) {
        const double t = row_of(v[k], r);
        if (lane == k) xp = t;
      }
      xp *= ir;
#pragma unroll
      for (int k = 0; k < decltype(slots)::value; ++k) {
        const double xr = __shfl_sync(0xffffffffu, xp, k);
#pragma unroll
        for (int s = 0; s < S; ++s) {
          const double y = s == 0 || r > 32 ? fma(-ur[s], xr, v[k][s]) : v[k][s];
          v[k][s] = lane + 32 * s == r ? xr : y;
        }
      }
    }
  };
  if (held > 4) back(std::integral_constant<int, KC>{});
  else if (held > 3) back(std::integral_constant<int, 4>{});
  else if (held > 2) back(std::integral_constant<int, 3>{});
  else if (held > 0) back(std::integral_constant<int, 2>{});
#pragma unroll
  for (int k = 0; k < KC; ++k) {
    const int c = c0 + 4 * k;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const int r = lane + 32 * s;
      if (r < M && c < tot) put(c - M, r, v[k][s]);
    }
  }
}

// Eliminates `nelim` nodes of a chain of `ntot` (local numbering; dir = -1: local node i is
// node base - i of the dim, else base + i).  MID: the chain is the middle, read from a.mid
// where the sides left it (from the band when there were no sides).  On return the W
// blocks and z of the eliminated nodes are in a.blocks and a.F; with nelim < ntot the
// window of the remaining nodes goes to `rest` ([hb M + 1][hb M], in the middle's own
// numbering).
template <int S, bool MID>
__device__ __forceinline__ void ts_eliminate(const TsArgs& a, int base, int dir, int nelim, int ntot, double* rest,
                                             bool rest_reversed, double* sm, unsigned rank, unsigned nc,
                                             cg::cluster_group& cluster) {
  const int M = a.M, hb = a.hb, nb = 2 * hb + 1, tid = threadIdx.x;
  const int MM = M * M;
  const TsLayout L = ts_layout(hb, M, (int)nc);
  const int rows = L.rows, cw = L.cw;
  double* win = sm + L.win;
  double* rhs = sm + L.rhs;
  double* wbuf = sm + L.wbuf;
  const bool has_rhs = rank == nc - 1;
  const bool from_mid = MID && a.nlo + a.nhi > 0;
  const int hM = hb * M, nring = hb + 1;
  const int step = (int)nc, sh = __ffs((int)nc) - 1;   // nc is a power of two
  const TsDiv byM(M), bycw(cw), byhM(hM);
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  auto first_own = [&](int g) { return g + (((int)rank - g) & (step - 1)); };   // smallest own column >= g
  auto count_own = [&](int g0, int end) { return g0 < end ? ((end - 1 - g0) >> sh) + 1 : 0; };
  auto wrap = [](int x, int m) { return x >= m ? x - m : x; };
  auto node_addr = [&](int i, int j, int m, int c) {   // A(i, j)[m][c] in the band
    const int gi = base + dir * i;
    return a.blocks + ((size_t)gi * nb + (dir * (j - i) + hb)) * MM + m * M + c;
  };
  // one entry of the chain's matrix into shared memory.  The high side leaves the middle's
  // own entries to the low side: it holds only its updates there.
  auto fetch = [&](double* dst, int i, int j, int m, int c) {
    if (MID && from_mid) {
      const double* lo = a.mid + (size_t)(j * M + c) * hM + (i * M + m);
      double v = __ldcg(lo);
      if (a.nhi > 0) v += __ldcg(lo + (size_t)(hM + 1) * hM);
      *dst = v;
    } else if (!MID && dir < 0 && i >= nelim && j >= nelim) {
      *dst = 0.0;
    } else {
      ts_copy8(dst, node_addr(i, j, m, c));
    }
  };
  auto fetch_rhs = [&](double* dst, int i, int m) {
    if (MID && from_mid) {
      const double* lo = a.mid + (size_t)hM * hM + (i * M + m);
      double v = __ldcg(lo);
      if (a.nhi > 0) v += __ldcg(lo + (size_t)(hM + 1) * hM);
      *dst = v;
    } else if (!MID && dir < 0 && i >= nelim) {
      *dst = 0.0;
    } else {
      ts_copy8(dst, a.F + (size_t)(base + dir * i) * M + m);
    }
  };
  // ---- the first window: panel of node 0 in every CTA, own columns of nodes 1 ..
  const int w0 = min(hb, ntot - 1);   // nodes after node 0 in the window
  for (int e = tid; e < M * (w0 + 1) * M; e += TS_THREADS) {
    const int r = byM.div(e), c = e - r * M, i = byM.div(r);
    fetch(sm + L.pan + (size_t)c * rows + r, i, 0, r - i * M, c);
  }
  {
    const int g0 = first_own(M), cnt = count_own(g0, (w0 + 1) * M), wr = (w0 + 1) * M;
    const TsDiv bywr(wr);
    for (int e = tid; e < cnt * wr; e += TS_THREADS) {
      const int ci = bywr.div(e), r = e - ci * wr, g = g0 + (ci << sh), i = byM.div(r), j = byM.div(g);
      fetch(win + (size_t)bycw.mod(g >> sh) * rows + r, i, j, r - i * M, g - j * M);
    }
  }
  if (has_rhs)
    for (int r = tid; r < (w0 + 1) * M; r += TS_THREADS) fetch_rhs(rhs + r, byM.div(r), byM.mod(r));
  ts_commit();
  ts_wait<0>();
  __syncthreads();

  int kring = 0, kpan = 0;   // k mod (hb + 1), k mod 3
  for (int k = 0; k < nelim; ++k) {
    const int nfol = min(hb, ntot - 1 - k);       // nodes after k in the window
    const int fr = nfol * M;                       // their rows
    const bool last = k == nelim - 1;
    const int enter = k + 1 + hb;                  // the node that enters the window
    const bool entering = !last && enter < ntot;
    // three panels: a CTA still updating with node k - 1's may already receive node k + 1's
    // from one that has passed the barrier in between
    double* pan = sm + L.pan + (size_t)kpan * M * rows;
    kpan = wrap(kpan + 1, 3);
    double* npan = sm + L.pan + (size_t)kpan * M * rows;
    const int lo = (k + 1) * M, g0 = first_own(lo), ncol = count_own(g0, lo + fr);
    const int nall = ncol + (has_rhs ? 1 : 0);
    const int s0 = bycw.mod(g0 >> sh);             // slot of the first own column
    auto column = [&](int ci) { return ci < ncol ? win + wrap(s0 + ci, cw) * rows : rhs; };
    auto ring_row = [&](int r) {                   // following row r in the ring
      const int i = byM.div(r);
      return wrap(kring + 1 + i, nring) * M + r - i * M;
    };
    if (warp < 4) {
      // ---- W = D^-1 A(k, .) of the own columns (the right-hand side as one more)
      double v[TS_COLS / 4][S];
#pragma unroll
      for (int q = 0; q < TS_COLS / 4; ++q)
#pragma unroll
        for (int s = 0; s < S; ++s) v[q][s] = 0.0;
#pragma unroll
      for (int q = 0; q < TS_COLS / 4; ++q) {
        const int c = 4 * q + warp;
        if (c >= M + nall) break;
        const double* x = c < M ? pan + c * rows : column(c - M) + kring * M;
#pragma unroll
        for (int s = 0; s < S; ++s)
          if (lane + 32 * s < M) v[q][s] = x[lane + 32 * s];
      }
      __syncthreads();
      ts_solve_node<S>(v, M, nall, sm + L.col, pan, rows, a.status, rank == 0, [&](int ci, int m, double w) {
        const int g = g0 + (ci << sh);
        wbuf[ci * M + m] = w;
        if (ci < ncol) *const_cast<double*>(node_addr(k, byM.div(g), m, byM.mod(g))) = w;
        else a.F[(size_t)(base + dir * k) * M + m] = w;
      });
    } else {
      // ---- meanwhile: the entries of the entering node
      __syncthreads();   // node k's rows of the window are in registers: their slots are free
      if (entering) {
        const int t4 = tid - 128;
        // its rows in the next panel: every CTA its own copy
        for (int e = t4; e < MM; e += 128) {
          const int m = byM.div(e), c = e - m * M;
          fetch(npan + (size_t)c * rows + hM + m, enter, k + 1, m, c);
        }
        const int h0 = first_own(lo + M), hn = count_own(h0, lo + M + hM), erow = kring * M;
        for (int e = t4; e < hn * M; e += 128) {   // its row of the own columns
          const int ci = byM.div(e), m = e - ci * M, g = h0 + (ci << sh), j = byM.div(g);
          fetch(win + (size_t)bycw.mod(g >> sh) * rows + erow + m, enter, j, m, g - j * M);
        }
        const int c0 = first_own(enter * M), cn = count_own(c0, (enter + 1) * M);
        for (int e = t4; e < cn * hM; e += 128) {   // its own columns (hb nodes follow k here)
          const int ci = byhM.div(e), r = e - ci * hM, g = c0 + (ci << sh), i = byM.div(r);
          fetch(win + (size_t)bycw.mod(g >> sh) * rows + ring_row(r), k + 1 + i, enter, r - i * M, g - enter * M);
        }
        if (has_rhs)
          for (int m = t4; m < M; m += 128) fetch_rhs(rhs + erow + m, enter, m);
      }
      ts_commit();
    }
    __syncthreads();
    // ---- A(i, .) -= A(i, k) W over the following nodes; the next panel's columns first,
    // pushed to every CTA: they and the entering rows are what the others wait for
    const int npush = last ? 0 : count_own(g0, lo + M) * fr;
    bool arrived = false;
    if (fr > 0) {
      const TsDiv byfr = fr == hM ? byhM : TsDiv(fr);
      for (int e0 = 0; e0 < nall * fr; e0 += TS_THREADS) {
        if (!arrived && e0 >= npush) {
          ts_arrive();
          arrived = true;
        }
        const int e = e0 + tid;
        if (e < nall * fr) {
          const int ci = byfr.div(e), r = e - ci * fr;
          double* x = column(ci) + ring_row(r);
          const double* p = pan + M + r;   // row r of the following nodes
          const double* wv = wbuf + ci * M;
          // the products' sum first, one subtraction after: a chain that starts from the entry
          // rounds at the entry's size in every term (2 - 3 times the error on ill-conditioned
          // systems)
          double sum = 0.0;
#pragma unroll 4
          for (int l = 0; l < M; ++l, p += rows) sum = fma(p[0], wv[l], sum);
          const double t0 = *x - sum;
          if (e < npush) {
            double* dst = npan + (size_t)(g0 + (ci << sh) - lo) * rows + r;
            for (unsigned t = 0; t < nc; ++t) *cluster.map_shared_rank(dst, t) = t0;
          } else {
            *x = t0;
          }
        }
        __syncwarp();
      }
    }
    if (!arrived) ts_arrive();
    ts_wait<0>();
    __syncthreads();
    ts_cluster_wait();
    kring = wrap(kring + 1, nring);
  }
  if (nelim < ntot) {
    // the remaining hb nodes, in the middle's numbering, column-major
    const int lo = nelim * M, g0 = first_own(lo), ncol = count_own(g0, ntot * M);
    const int nall = ncol + (has_rhs ? 1 : 0), nr = ntot * M - lo;
    const TsDiv bynr(nr);
    for (int e = tid; e < nall * nr; e += TS_THREADS) {
      const int ci = bynr.div(e), r = e - ci * nr, il = byM.div(r), m = r - il * M;
      const int mi = rest_reversed ? hb - 1 - il : il, row = wrap(kring + il, nring) * M + m;
      if (ci < ncol) {
        const int g = g0 + (ci << sh), j = byM.div(g), jl = j - nelim;
        const int mj = rest_reversed ? hb - 1 - jl : jl;
        rest[(size_t)(mj * M + g - j * M) * hM + mi * M + m] = win[(size_t)bycw.mod(g >> sh) * rows + row];
      } else {
        rest[(size_t)hM * hM + mi * M + m] = rhs[row];
      }
    }
  }
}

// Clusters 0 and 1: the low and the high end.
template <int S>
__global__ void __launch_bounds__(TS_THREADS) ts_sides_kernel(TsArgs a) {
  extern __shared__ __align__(16) double ts_smem[];
  cg::cluster_group cluster = cg::this_cluster();
  const unsigned nc = cluster.num_blocks(), rank = cluster.block_rank();
  const int side = blockIdx.x / nc;
  taps_pdl_wait();
  cluster.sync();   // every CTA of the cluster runs before its shared memory is written
  if (side == 0)
    ts_eliminate<S, false>(a, 0, 1, a.nlo, a.nlo + a.nmid, a.mid, false, ts_smem, rank, nc, cluster);
  else
    ts_eliminate<S, false>(a, a.n - 1, -1, a.nhi, a.nhi + a.nmid,
                           a.mid + (size_t)(a.hb * a.M + 1) * a.hb * a.M, true, ts_smem, rank, nc, cluster);
}

// x_k = z_k - sum_j W(k, k + dir j) x_{k + dir j} along a chain of nodes k0, k0 - dir, ...
// (count nodes), the first with `have` following nodes, then one more each up to hb.  The W
// blocks of the next nodes are in flight, laid out [m][following node, mode]; xs holds the
// last hb + 1 nodes' x twice over, so that any hb consecutive ones lie in a row.  Eight lanes
// share an output's dot product.  X is written for the nodes from index `write_from` on.
__device__ __forceinline__ void ts_backsub(const TsArgs& a, int k0, int dir, int count, int have, int write_from,
                                           double* xs, double* buf, int stages) {
  const int M = a.M, hb = a.hb, nb = 2 * hb + 1, tid = threadIdx.x, MM = M * M, hM = hb * M, nring = hb + 1;
  const int stage = hM * M + M;
  const TsDiv byM(M), byMM(MM), byring(nring);
  auto load = [&](int t, double* d) {
    if (t < count) {
      const int k = k0 - dir * t, nf = min(hb, have + t);
      // blocks k+1 .. k+nf (dir 1) lie one after another; k-1 .. k-nf (dir -1) too, downwards
      const double* w = a.blocks + ((size_t)k * nb + (dir > 0 ? hb + 1 : hb - nf)) * MM;
      for (int e = tid - 128; e < nf * MM; e += 128) {
        const int jj = byMM.div(e), rem = e - jj * MM, m = byM.div(rem);
        ts_copy8(d + m * hM + jj * M + rem - m * M, w + e);
      }
      for (int m = tid - 128; m < M; m += 128) ts_copy8(d + hM * M + m, a.F + (size_t)k * M + m);
    }
    ts_commit();
  };
  const bool loads = __shfl_sync(0xffffffffu, tid >> 5, 0) >= 4;   // four warps load, four compute
  if (loads)
    for (int t = 0; t < stages - 1; ++t) load(t, buf + t * stage);
  int cur = 0;
  for (int t = 0; t < count; ++t) {
    // at most stages - 2 younger groups may still be in flight
    if (stages >= 4) ts_wait<2>();
    else if (stages == 3) ts_wait<1>();
    else ts_wait<0>();
    __syncthreads();   // node t's blocks and the previous node's x
    if (loads) load(t + stages - 1, buf + (cur == 0 ? stages - 1 : cur - 1) * stage);
    const int k = k0 - dir * t, nf = min(hb, have + t);
    const double* d = buf + cur * stage;
    const double* xw = xs + byring.mod(dir > 0 ? k + 1 : k - nf) * M;
    for (int o = loads ? M * 8 + 31 : tid; o < ((M * 8 + 31) & ~31); o += 128) {
      const int m = o >> 3, part = o & 7;
      double s0 = 0.0;
      if (m < M) {
        const double* wr = d + m * hM;
#pragma unroll 4
        for (int c = part; c < nf * M; c += 8) s0 = fma(wr[c], xw[c], s0);
      }
      s0 += __shfl_xor_sync(0xffffffffu, s0, 4);
      s0 += __shfl_xor_sync(0xffffffffu, s0, 2);
      s0 += __shfl_xor_sync(0xffffffffu, s0, 1);
      if (part == 0 && m < M) {
        const double x = d[hM * M + m] - s0;
        double* xo = xs + byring.mod(k) * M + m;
        xo[0] = x;
        xo[nring * M] = x;
        if (t >= write_from) {
          if (!isfinite(x)) taps_flag(a.status, TAPS_DEV_NONFINITE);
          a.X[(size_t)m * a.n + k] = x;
        }
      }
    }
    if (++cur == stages) cur = 0;
  }
  ts_wait<0>();
  __syncthreads();
}

// One cluster: the middle, then CTA 0 substitutes back from the middle to the low end and
// CTA 1 (CTA 0 itself in a cluster of one) from the middle to the high end.
template <int S>
__global__ void __launch_bounds__(TS_THREADS) ts_finish_kernel(TsArgs a, int stages) {
  extern __shared__ __align__(16) double ts_smem[];
  cg::cluster_group cluster = cg::this_cluster();
  const unsigned nc = cluster.num_blocks(), rank = cluster.block_rank();
  taps_pdl_wait();
  if (a.Save) {
    const long long tot = (long long)a.n * a.M;
    for (long long e = rank * TS_THREADS + threadIdx.x; e < tot; e += (long long)nc * TS_THREADS) a.Save[e] = a.X[e];
  }
  cluster.sync();
  ts_eliminate<S, true>(a, a.nlo, 1, a.nmid, a.nmid, nullptr, false, ts_smem, rank, nc, cluster);
  // the W blocks and z the other CTAs wrote
  __threadfence();
  cluster.sync();
  double* xs = ts_smem;                              // [2][(hb + 1) M]: solved nodes
  double* buf = ts_smem + 2 * ts_layout(a.hb, a.M, (int)nc).rows;
  if (rank == 0) ts_backsub(a, a.nlo + a.nmid - 1, 1, a.nlo + a.nmid, 0, 0, xs, buf, stages);
  if (a.nhi > 0 && rank == (nc > 1 ? 1u : 0u)) {
    ts_backsub(a, a.nlo + a.nmid - 1, 1, a.nmid, 0, a.nmid, xs, buf, stages);   // the middle again, not written
    ts_backsub(a, a.nlo + a.nmid, -1, a.nhi, a.hb, 0, xs, buf, stages);
  }
}

// ---------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------
static size_t ts_smem_bytes(int hb, int M, int nc) { return sizeof(double) * ts_layout(hb, M, nc).total; }

static bool ts_fits(int hb, int M, int nc, size_t smem) {
  return M + ts_layout(hb, M, nc).cw + 1 <= TS_COLS && ts_smem_bytes(hb, M, nc) <= smem;
}

// CTAs per cluster: the largest the device places, unless a CTA would hold fewer than four
// of the window's columns.  Measured per solve (elimination, middle, back substitution, us,
// 64 nodes, hb = 5) with 4 / 8 / 16 CTAs: M = 6: 219 / 194 / 187, M = 10: 398 / 303 / 266,
// M = 20: 1731 / 958 / 696, M = 30: - / 2573 / 1372; 14 nodes, M = 4: 56 / 54 / 54.
static int ts_cluster_size(int hb, int M, int most) {
  int nc = 1;
  while (nc < most && (hb + 1) * M > 4 * nc) nc *= 2;
  return nc;
}

static cudaError_t ts_launch(void (*fn)(TsArgs), int grid, int nc, size_t smem, cudaStream_t s, const TsArgs& a) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(TS_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = nc;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, fn, a);
}
static cudaError_t ts_launch_finish(void (*fn)(TsArgs, int), int nc, size_t smem, cudaStream_t s, const TsArgs& a,
                                    int stages) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nc);
  cfg.blockDim = dim3(TS_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = nc;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, fn, a, stages);
}

// Largest cluster (16, 8, ... or 0: none) that the device can place with `smem` bytes.
static int ts_most_ctas(const void* fn, size_t smem) {
  for (int nc = 16; nc >= 1; nc /= 2) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nc);
    cfg.blockDim = dim3(TS_THREADS);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = nc;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg) == cudaSuccess && clusters > 0) return nc;
    cudaGetLastError();
  }
  return 0;
}

// Shared-memory and cluster-size opt-in; *most: the largest cluster with the whole of a
// CTA's shared memory, *smem that memory.
int taps_ts_setup(int maxsm, int* most, size_t* smem) {
  const void* fns[4] = {(const void*)ts_sides_kernel<1>, (const void*)ts_sides_kernel<2>,
                        (const void*)ts_finish_kernel<1>, (const void*)ts_finish_kernel<2>};
  *most = 16;
  *smem = (size_t)maxsm;
  for (const void* fn : fns) {
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) cudaGetLastError();
    TAPS_TRY(taps_allow_dyn_smem(fn, maxsm));
    cudaFuncAttributes fa;
    TAPS_CUDA(cudaFuncGetAttributes(&fa, fn));
    *smem = std::min(*smem, (size_t)maxsm - fa.sharedSizeBytes);
    *most = std::min(*most, ts_most_ctas(fn, (size_t)maxsm - fa.sharedSizeBytes));
  }
  return TAPS_OK;
}

// CTAs per cluster for a dim of half-bandwidth hb at M modes; 0: the one-ended route.
// Beyond hb = 5 (s >= 3) the one-ended elimination stays, to keep the results that users of
// those spaces have: not for accuracy (backward errors of single solves, 32 nodes, 6 and 12 modes
// with two of them 1e-5 apart, from both ends / from one: s = 2: 7.2e-14, 1.5e-13 / 8.4e-14,
// 1.1e-13; s = 3: 9.1e-14, 1.0e-13 / 8.6e-14, 1.3e-13) nor for speed (64 nodes of 10 modes at
// s = 3: 301 us / 1240 us), but because fixed-M iterations at third order end where rounding takes
// them, and the order that the space-time refinement study shows at s = p = 3 depends on it.
int taps_ts_ctas(const taps_problem* P, int hb, int M) {
  if (hb > 5 || M > 64 || P->ts_most < 1) return 0;
  int nc = ts_cluster_size(hb, M, P->ts_most);
  while (nc < P->ts_most && !ts_fits(hb, M, nc, P->ts_maxsm)) nc *= 2;
  return ts_fits(hb, M, nc, P->ts_maxsm) ? nc : 0;
}

size_t taps_ts_scratch_doubles(int hb, int M) { return 2 * ((size_t)hb * M + 1) * hb * M; }

// Solves the reduced system of dim d assembled in P->d_blocks / P->d_F; the factor before
// the solve goes to P->d_Uold.  The profile counts the ends' kernel (with the elimination's flops
// and the bytes) and the middle's apart.
int taps_ts_solve(taps_problem* P, taps_factors* U, int d, int nc, double lu_flops, double bs_flops, double bytes) {
  const taps_dim* dm = P->dims[d];
  TsArgs a;
  memset(&a, 0, sizeof(a));
  a.blocks = P->d_blocks;
  a.F = P->d_F;
  a.mid = P->d_ts;
  a.n = dm->nf;
  a.hb = dm->hb;
  a.M = U->M;
  a.nmid = std::min(a.n, a.hb);
  a.nlo = (a.n - a.nmid + 1) / 2;
  a.nhi = a.n - a.nmid - a.nlo;
  a.X = U->d_U[d];
  a.Save = P->d_Uold;
  a.status = P->d_status;
  const bool wide = a.M > 32;
  size_t smem = ts_smem_bytes(a.hb, a.M, nc);
  const bool ends = a.nlo > 0;
  if (ends) {
    const int tk = prof_begin(P, TAPS_PROF_BLOCK_ENDS);
    const cudaError_t ce = ts_launch(wide ? ts_sides_kernel<2> : ts_sides_kernel<1>, (a.nhi > 0 ? 2 : 1) * nc, nc, smem,
                                     P->stream, a);
    if (ce != cudaSuccess) {
      taps_note_cuda_error(ce, "two-sided elimination launch", __FILE__, __LINE__);
      return TAPS_ERR_CUDA;
    }
    prof_end(P, TAPS_PROF_BLOCK_ENDS, tk, lu_flops, bytes);
  }
  // the back substitution's stages share the elimination's shared memory
  const size_t rows = 2 * (size_t)(a.hb + 1) * a.M, stage = (size_t)a.hb * a.M * a.M + a.M;
  int stages = TS_STAGES;
  while (stages > 2 && sizeof(double) * (rows + stages * stage) > std::max(smem, (size_t)P->ts_maxsm / 2)) --stages;
  smem = std::max(smem, sizeof(double) * (rows + stages * stage));
  const int fnc = std::max(nc, std::min(2, P->ts_most));
  smem = std::max(smem, ts_smem_bytes(a.hb, a.M, fnc));
  const int tk = prof_begin(P, TAPS_PROF_BLOCK_LU);
  const cudaError_t ce =
      ts_launch_finish(wide ? ts_finish_kernel<2> : ts_finish_kernel<1>, fnc, smem, P->stream, a, stages);
  if (ce != cudaSuccess) {
    taps_note_cuda_error(ce, "middle and back substitution launch", __FILE__, __LINE__);
    return TAPS_ERR_CUDA;
  }
  prof_end(P, TAPS_PROF_BLOCK_LU, tk, ends ? bs_flops : lu_flops + bs_flops, ends ? 0.0 : bytes);
  return TAPS_OK;
}
