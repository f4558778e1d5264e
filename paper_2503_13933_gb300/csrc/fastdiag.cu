// Fast-diagonalisation reduced solver (Sec. 2.6: the subspace system of one dimension
// is a generalised Sylvester equation, solved by fast diagonalisation).
//
// For a dimension whose distinct operators form a symmetric-definite pencil (A, B)
// (e.g. stiffness K and mass M; or a single SPD operator B, A = 0), the pencil is
// diagonalised once: Phi^T B Phi = I, Phi^T A Phi = diag(mu).  The reduced system
//     A U C_A^T + B U C_B^T = F        (U: n x M, C: M x M, possibly nonsymmetric)
// becomes, with U = Phi Y and G = Phi^T F, n independent M x M systems
//     (mu_i C_A + C_B) Y[i,:]^T = G[i,:]^T,
// so a solve costs two n x n x M products and n small LU solves instead of a
// sequential block elimination over the n block rows.
//
// The one-off pencil decomposition, in FP64: banded Cholesky B = L L^T on one warp,
// S = L^{-1} A L^{-T} (one thread per column), Householder tridiagonalisation S = Q T Q^T on
// one thread-block cluster or on all SMs; then, in parallel, the eigenvalues of T by
// Sturm-count multisection (one warp per eigenvalue), its eigenvectors by inverse iteration
// (one thread per eigenvector, one per cluster of nearly equal eigenvalues), one step of
// symmetric orthogonalisation, the back-transform Z = Q Z_T (one warp per column), and
// Phi = L^{-T} Z (one thread per column).
#include <string.h>

#include <algorithm>

#include <cooperative_groups.h>

#include "small_lu.cuh"
#include "taps_internal.cuh"

#define FD_THREADS 1024

__global__ void fd_dense_kernel(const double* __restrict__ bandA, const double* __restrict__ bandB, int n,
                                int hb, double* __restrict__ A, double* __restrict__ B) {
  long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)n * n) return;
  int i = idx / n, j = idx % n, k = j - i + hb, nb = 2 * hb + 1;
  bool in = (k >= 0 && k < nb);
  A[idx] = (bandA && in) ? bandA[(size_t)i * nb + k] : 0.0;
  B[idx] = in ? bandB[(size_t)i * nb + k] : 0.0;
}

// Banded Cholesky B = L L^T (lower factor in place in the dense B; half-bandwidth hb) and the
// reciprocals of L's diagonal, by one warp with the band in shared memory: a column is a chain
// of a square root, a division and an update, and more threads only add barriers to it (1024
// threads, three block barriers a column: 394 us for 254 nodes).
__global__ void __launch_bounds__(32) fd_cholesky_kernel(const double* __restrict__ band, double* B, int n, int hb,
                                                         double* __restrict__ linv, int* status) {
  extern __shared__ double Lb[];   // [n][hb + 1]: entry (i, i - t) at t
  const int lane = threadIdx.x, W = hb + 1, nb = 2 * hb + 1;
  for (int idx = lane; idx < n * W; idx += 32) {
    const int i = idx / W, t = idx - i * W;
    Lb[idx] = i - t >= 0 ? band[(size_t)i * nb + hb - t] : 0.0;
  }
  __syncwarp();
  for (int k = 0; k < n; ++k) {
    double piv = Lb[k * W];
    if (!(piv > 0.0) || !isfinite(piv)) {
      if (lane == 0) taps_flag(status, TAPS_DEV_SINGULAR);
      piv = 1.0;
    }
    const double lkk = sqrt(piv);
    const int w = min(n - 1, k + hb) - k;
    __syncwarp();
    if (lane == 0) Lb[k * W] = lkk;
    if (lane >= 1 && lane <= w) Lb[(k + lane) * W + lane] /= lkk;
    __syncwarp();
    for (int idx = lane; idx < w * w; idx += 32) {
      const int x = 1 + idx / w, y = 1 + idx % w;   // rows k + x >= columns k + y
      if (y <= x) {
        double* e = Lb + (k + x) * W + (x - y);
        *e -= Lb[(k + x) * W + x] * Lb[(k + y) * W + y];
      }
    }
    __syncwarp();
  }
  for (int idx = lane; idx < n * W; idx += 32) {
    const int i = idx / W, t = idx - i * W;
    if (i - t >= 0) B[(size_t)i * n + i - t] = Lb[idx];
    if (t == 0) linv[i] = taps_rcp(Lb[idx]);
  }
}

// The same for a band that does not fit one CTA's shared memory.
__global__ void __launch_bounds__(FD_THREADS) fd_cholesky_global_kernel(double* B, int n, int hb,
                                                                        double* __restrict__ linv, int* status) {
  const int tid = threadIdx.x, nt = blockDim.x;
#define AT(M_, i, j) M_[(size_t)(i) * n + (j)]
  for (int k = 0; k < n; ++k) {
    if (tid == 0) {
      double piv = AT(B, k, k);
      if (!(piv > 0.0) || !isfinite(piv)) {
        taps_flag(status, TAPS_DEV_SINGULAR);
        piv = 1.0;
      }
      AT(B, k, k) = sqrt(piv);
    }
    __syncthreads();
    double lkk = AT(B, k, k);
    if (tid == 0) linv[k] = taps_rcp(lkk);
    int top = min(n - 1, k + hb);
    for (int i = k + 1 + tid; i <= top; i += nt) AT(B, i, k) /= lkk;
    __syncthreads();
    int w = top - k;
    for (int idx = tid; idx < w * w; idx += nt) {
      int i = k + 1 + idx / w, j = k + 1 + idx % w;
      if (j <= i) AT(B, i, j) -= AT(B, i, k) * AT(B, j, k);
    }
    __syncthreads();
  }
#undef AT
}

// Out[:, c] = L^{-1} (In[:, c] or, with transposed input, In[c, :]^T) for the banded
// lower factor L (half-bandwidth HB): one thread per column c, the chain of n
// substitutions with the diagonal's reciprocals; 32-thread CTAs spread the columns over
// the SMs.  The last HB values stay in registers and the factor's rows are loaded FD_AHEAD
// rows early, so a step is its HB + 1 FP64 instructions (read back from memory, with a
// reciprocal per step and column: 248 us for 254 nodes).
#define FD_AHEAD 4
template <int HB>
__global__ void __launch_bounds__(32) fd_lsolve_kernel(const double* __restrict__ L, const double* __restrict__ linv,
                                                       const double* __restrict__ In, int n, int trans_in,
                                                       double* __restrict__ Out) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n) return;
  double x[HB];                                   // values of rows i - HB .. i - 1
  double l[FD_AHEAD][HB], in[FD_AHEAD], li[FD_AHEAD];
  auto load = [&](int i, double (&p)[HB], double& q, double& r) {
    if (i >= n) return;
#pragma unroll
    for (int t = 0; t < HB; ++t) p[t] = i - HB + t >= 0 ? L[(size_t)i * n + i - HB + t] : 0.0;
    q = trans_in ? In[(size_t)c * n + i] : In[(size_t)i * n + c];
    r = linv[i];
  };
#pragma unroll
  for (int t = 0; t < HB; ++t) x[t] = 0.0;
#pragma unroll
  for (int a = 0; a < FD_AHEAD; ++a) load(a, l[a], in[a], li[a]);
  for (int i0 = 0; i0 < n; i0 += FD_AHEAD) {
#pragma unroll
    for (int a = 0; a < FD_AHEAD; ++a) {
      const int i = i0 + a;
      if (i >= n) break;
      double s = in[a];
#pragma unroll
      for (int t = 0; t < HB; ++t)
        if (i - HB + t >= 0) s -= l[a][t] * x[t];
      s = s * li[a];
      Out[(size_t)i * n + c] = s;
#pragma unroll
      for (int t = 0; t + 1 < HB; ++t) x[t] = x[t + 1];
      x[HB - 1] = s;
      load(i + FD_AHEAD, l[a], in[a], li[a]);
    }
  }
}

// A = (V + V^T) / 2
__global__ void fd_symmetrize_kernel(const double* __restrict__ V, int n, double* __restrict__ A) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)n * n) return;
  const int i = (int)(idx / n), j = (int)(idx % n);
  A[idx] = 0.5 * (V[(size_t)i * n + j] + V[(size_t)j * n + i]);
}

// ---------------------------------------------------------------------------------
// Householder tridiagonalisation S = Q T Q^T of the symmetric S held in A (n x n,
// row-major), on one cluster of NC CTAs (16 where the GPU can place a 16-CTA cluster,
// else 8; the arithmetic is the same for both) with hardware cluster barriers between
// the phases of a step.  Step k: every CTA stages column k below the diagonal in
// shared memory and forms the same reflector v (beta = 2 / v.v); one warp per row of
// the cluster computes p = beta S22 v; after a cluster barrier every CTA forms
// w = p - (beta v.p / 2) v and its warps update their rows of S22 -= v w^T + w v^T;
// a second barrier ends the step.  Values written by other CTAs are read through L2.
// On exit (d, e) hold T (e[i] couples i and i+1), the rows of V the reflectors
// (row k: entries k+1 .. n-1) and beta their factors.
// ---------------------------------------------------------------------------------
#define TD_THREADS 1024
#define TDS_THREADS 512    // S in distributed shared memory: about a warp per row and CTA
__device__ __forceinline__ void td_cluster_sync() {
  asm volatile(
      "barrier.cluster.arrive.release.aligned;\n\t"
      "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <int NC>
__global__ void __launch_bounds__(TD_THREADS)
    fd_tridiag_kernel(double* __restrict__ A, double* __restrict__ V, double* __restrict__ p,
                      double* __restrict__ beta, double* __restrict__ d, double* __restrict__ e, int n) {
  extern __shared__ double tds[];   // v [n], p [n], w [n]
  __shared__ double red[32];
  double* vs = tds;
  double* ps = tds + n;
  double* ws = tds + 2 * n;
  const int rank = blockIdx.x;   // the grid is one cluster
  const int tid = threadIdx.x, lane = tid & 31;
  const int gwarp = rank * (TD_THREADS / 32) + (tid >> 5);
  const int nwarps = NC * (TD_THREADS / 32);
#define AT(i, j) A[(size_t)(i) * n + (j)]
  for (int k = 0; k + 2 < n; ++k) {
    const int len = n - k - 1;
    double s2 = 0.0;
    for (int t = tid; t < len; t += TD_THREADS) {
      const double x = __ldcg(&AT(k + 1 + t, k));
      vs[t] = x;
      s2 += x * x;
    }
    s2 = block_sum(s2, red);   // also orders the vs writes
    if (s2 == 0.0) {           // the same in every CTA: nothing to reflect
      if (rank == 0 && tid == 0) {
        beta[k] = 0.0;
        d[k] = __ldcg(&AT(k, k));
        e[k] = 0.0;
      }
      continue;
    }
    const double x0 = vs[0];
    const double alpha = -copysign(sqrt(s2), x0);
    const double v0 = x0 - alpha;
    const double bk = 2.0 / (s2 - x0 * x0 + v0 * v0);
    __syncthreads();
    if (tid == 0) vs[0] = v0;
    __syncthreads();
    // p = beta S22 v, one warp per row
    for (int i = gwarp; i < len; i += nwarps) {
      const double* row = A + (size_t)(k + 1 + i) * n + (k + 1);
      double acc = 0.0;
      for (int t = lane; t < len; t += 32) acc += __ldcg(row + t) * vs[t];
      acc = warp_sum(acc);
      if (lane == 0) p[i] = bk * acc;
    }
    td_cluster_sync();
    double pv = 0.0;
    for (int t = tid; t < len; t += TD_THREADS) {
      const double pt = __ldcg(p + t);
      ps[t] = pt;
      pv += pt * vs[t];
    }
    pv = block_sum(pv, red);
    const double Kc = 0.5 * bk * pv;
    for (int t = tid; t < len; t += TD_THREADS) ws[t] = ps[t] - Kc * vs[t];
    __syncthreads();
    for (int i = gwarp; i < len; i += nwarps) {
      double* row = A + (size_t)(k + 1 + i) * n + (k + 1);
      const double vi = vs[i], wi = ws[i];
      for (int t = lane; t < len; t += 32) row[t] = __ldcg(row + t) - (vi * ws[t] + wi * vs[t]);
    }
    if (rank == 0) {
      for (int t = tid; t < len; t += TD_THREADS) V[(size_t)k * n + k + 1 + t] = vs[t];
      if (tid == 0) {
        beta[k] = bk;
        d[k] = __ldcg(&AT(k, k));
        e[k] = alpha;
      }
    }
    td_cluster_sync();
  }
  if (rank == 0 && tid == 0) {
    if (n >= 2) {
      d[n - 2] = __ldcg(&AT(n - 2, n - 2));
      e[n - 2] = __ldcg(&AT(n - 1, n - 2));
    }
    d[n - 1] = __ldcg(&AT(n - 1, n - 1));
    e[n - 1] = 0.0;
    for (int k = (n >= 2 ? n - 2 : 0); k < n; ++k) beta[k] = 0.0;
  }
#undef AT
}

// The same tridiagonalisation with S held in the cluster's distributed shared memory
// (n small enough that ceil(n / NC) rows of n doubles fit one CTA's shared memory):
// CTA r keeps rows i = r, r + NC, ...  Step k: every CTA gathers column k from the
// rows' owners (remote shared-memory loads), forms the reflector, computes p_i for its
// own rows and stores each p_i into every CTA's copy of p; after a cluster barrier
// every CTA forms w and updates its own rows; a second barrier ends the step.  S never
// leaves shared memory.  Sums over the column run on the warps that hold entries of it and its
// scalars (square root, division) on one warp; every warp forming them was two thirds of a
// step (254 nodes: 3.51 -> 1.73 ms, the same bits: the other warps' summands were zeros).
template <int NC>
__global__ void __launch_bounds__(TDS_THREADS)
    fd_tridiag_dsmem_kernel(const double* __restrict__ A, double* __restrict__ V, double* __restrict__ beta,
                            double* __restrict__ d, double* __restrict__ e, int n) {
  extern __shared__ double tsm[];   // vs [n] | ps [n] | ws [n] | own rows [nr][n]
  __shared__ double red[32], sc[4];
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nwarps = TDS_THREADS / 32;
  double* vs = tsm;
  double* ps = tsm + n;
  double* ws = tsm + 2 * n;
  double* rows = tsm + 3 * n;
  const int nr = (n - rank + NC - 1) / NC;   // rows i = rank + NC * l, l < nr
  for (long long idx = tid; idx < (long long)nr * n; idx += TDS_THREADS) {
    const int l = (int)(idx / n), j = (int)(idx % n);
    rows[(size_t)l * n + j] = A[(size_t)(rank + NC * l) * n + j];
  }
  cluster.sync();
  for (int k = 0; k + 2 < n; ++k) {
    const int len = n - k - 1, nact = min((len + 31) / 32, nwarps);   // warps with entries of the column
    // column k below the diagonal, from the owners of its rows
    if (warp < nact) {
      double s2 = 0.0;
      for (int t = tid; t < len; t += TDS_THREADS) {
        const int i = k + 1 + t;
        const double* owner_rows = cluster.map_shared_rank(rows, i % NC);
        const double x = owner_rows[(size_t)(i / NC) * n + k];
        vs[t] = x;
        s2 += x * x;
      }
      s2 = warp_sum(s2);
      if (lane == 0) red[warp] = s2;
    }
    __syncthreads();
    if (warp == 0) {   // the column's scalars once: 32 warps forming them cost 32 times the issue
      const double s2 = warp_sum(lane < nact ? red[lane] : 0.0);
      if (lane == 0) {
        sc[0] = s2;
        if (s2 != 0.0) {
          const double x0 = vs[0];
          const double al = -copysign(sqrt(s2), x0);
          const double v0 = x0 - al;
          sc[1] = al;
          sc[2] = 2.0 / (s2 - x0 * x0 + v0 * v0);
          vs[0] = v0;
        }
      }
    }
    __syncthreads();
    if (sc[0] == 0.0) {   // the same in every CTA
      if (k % NC == rank && tid == 0) d[k] = rows[(size_t)(k / NC) * n + k];
      if (rank == 0 && tid == 0) {
        beta[k] = 0.0;
        e[k] = 0.0;
      }
      cluster.sync();
      continue;
    }
    const double alpha = sc[1], bk = sc[2];
    // p_i for own rows i >= k + 1, pushed into every CTA's ps
    const int l0 = (k + 1 - rank + NC - 1) / NC;   // first own row >= k + 1
    for (int l = l0 + warp; l < nr; l += nwarps) {
      const int i = rank + NC * l;
      const double* row = rows + (size_t)l * n + (k + 1);
      double acc = 0.0;
      for (int t = lane; t < len; t += 32) acc += row[t] * vs[t];
      acc = warp_sum(acc) * bk;
      if (lane < NC) cluster.map_shared_rank(ps, lane)[i - k - 1] = acc;
    }
    cluster.sync();
    if (warp < nact) {
      double pv = 0.0;
      for (int t = tid; t < len; t += TDS_THREADS) pv += ps[t] * vs[t];
      pv = warp_sum(pv);
      if (lane == 0) red[warp] = pv;
    }
    __syncthreads();
    if (warp == 0) {
      const double pv = warp_sum(lane < nact ? red[lane] : 0.0);
      if (lane == 0) sc[3] = 0.5 * bk * pv;
    }
    __syncthreads();
    if (warp < nact) {
      const double Kc = sc[3];
      for (int t = tid; t < len; t += TDS_THREADS) ws[t] = ps[t] - Kc * vs[t];
    }
    __syncthreads();
    for (int l = l0 + warp; l < nr; l += nwarps) {
      const int i = rank + NC * l - (k + 1);   // index within the trailing block
      double* row = rows + (size_t)l * n + (k + 1);
      const double vi = vs[i], wi = ws[i];
      for (int t = lane; t < len; t += 32) row[t] -= vi * ws[t] + wi * vs[t];
    }
    if (rank == 0) {
      for (int t = tid; t < len; t += TDS_THREADS) V[(size_t)k * n + k + 1 + t] = vs[t];
      if (tid == 0) {
        beta[k] = bk;
        e[k] = alpha;
      }
    }
    if (k % NC == rank && tid == 0) d[k] = rows[(size_t)(k / NC) * n + k];
    cluster.sync();
  }
  if (tid == 0) {
    for (int i = (n >= 2 ? n - 2 : 0); i < n; ++i)
      if (i % NC == rank) d[i] = rows[(size_t)(i / NC) * n + i];
    if (n >= 2 && (n - 1) % NC == rank) e[n - 2] = rows[(size_t)((n - 1) / NC) * n + (n - 2)];
    if (rank == 0) {
      e[n - 1] = 0.0;
      for (int k = (n >= 2 ? n - 2 : 0); k < n; ++k) beta[k] = 0.0;
    }
  }
}

// The same with the rows of S in the shared memory of the whole chip, one cooperative launch: CTA
// r keeps rows r, r + G, ...  One grid barrier per step: a pass over the own rows applies the last
// step's update, multiplies by the new reflector and publishes p and row k + 1 (the next column,
// before this step's update) in global memory; after the barrier every CTA forms w and the
// updated column from them, and from that the next reflector.  Two copies of the published
// vectors, so that a CTA ahead never overwrites what another still reads.  The chain of a step
// (barrier, two block sums, the reflector's scalars) is the bound; the cluster version reads and
// writes S in L2 twice a step on 16 SMs.  1534 nodes: 128 ms on a cluster, 21.7 ms here.
#define TDG_THREADS 512
#define TDG_PER 4   // entries of a column to a thread: n <= TDG_THREADS * TDG_PER
__global__ void __launch_bounds__(TDG_THREADS)
    fd_tridiag_grid_kernel(const double* __restrict__ A, double* __restrict__ V, double* __restrict__ beta,
                           double* __restrict__ d, double* __restrict__ e, int n, double* xch, unsigned* bar,
                           int* status) {
  extern __shared__ double tsm[];   // two reflectors [2][n] | w [n] | own rows [nr][n]
  __shared__ double red[TDG_THREADS / 32], sc[4];
  const int G = gridDim.x, rank = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = TDG_THREADS / 32;
  double *v = tsm, *vn = tsm + n, *ws = tsm + 2 * n, *rows = tsm + 3 * n;
  const int nr = rank < n ? (n - rank + G - 1) / G : 0;   // rows rank + G l, l < nr
  for (long long idx = tid; idx < (long long)nr * n; idx += TDG_THREADS) {
    const int l = (int)(idx / n), j = (int)(idx % n);
    rows[(size_t)l * n + j] = A[(size_t)(rank + G * l) * n + j];
  }
  double x[TDG_PER];   // row k from its diagonal on: entries tid + TDG_THREADS j
#pragma unroll
  for (int j = 0; j < TDG_PER; ++j) {
    const int t = tid + TDG_THREADS * j;
    x[j] = t < n ? A[t] : 0.0;
  }
  // sum over the block of one value per thread of the first `count`; warp 0 holds it
  auto partial_sum = [&](double y, int count) {
    if (warp * 32 < count) {
      y = warp_sum(y);
      if (lane == 0) red[warp] = y;
    } else if (lane == 0) {
      red[warp] = 0.0;
    }
    __syncthreads();
    return warp == 0 ? warp_sum(lane < nwarps ? red[lane] : 0.0) : 0.0;
  };
  // the reflector of step k from row k in x: vn, sc[1] = alpha, sc[2] = beta; zero for a zero column
  auto reflect = [&](int k) {
    const int len = n - k - 1;
    double s2 = 0.0;
#pragma unroll
    for (int j = 0; j < TDG_PER; ++j) {
      const int t = tid + TDG_THREADS * j;
      if (t >= 1 && t <= len) {
        vn[t - 1] = x[j];
        s2 = fma(x[j], x[j], s2);
      }
    }
    if (tid == 1) sc[3] = x[0];
    s2 = partial_sum(s2, len + 1);
    if (tid == 0) {
      double al = 0.0, v0 = 0.0, bk = 0.0;
      if (s2 != 0.0) {
        const double x0 = sc[3];
        al = -copysign(sqrt(s2), x0);
        v0 = x0 - al;
        bk = 2.0 / (s2 - x0 * x0 + v0 * v0);
      }
      vn[0] = v0;
      sc[1] = al;
      sc[2] = bk;
      if (rank == 0) {
        d[k] = x[0];
        e[k] = al;
        beta[k] = bk;
      }
    }
    __syncthreads();
    if (rank == 0)
      for (int t = tid; t < len; t += TDG_THREADS) V[(size_t)k * n + k + 1 + t] = vn[t];
  };
  reflect(0);   // its barriers also order the rows' loads
  for (int k = 0; k + 2 < n; ++k) {
    const int len = n - k - 1;
    const double bk = sc[2];
    double* pbuf = xch + (size_t)(k & 1) * 2 * n;
    double* rbuf = pbuf + n;
    for (int l = (k + 1 - rank + G - 1) / G + warp; l < nr; l += nwarps) {
      const int i = rank + G * l;
      double* row = rows + (size_t)l * n + (k + 1);
      const double vi = k > 0 ? v[i - k] : 0.0, wi = k > 0 ? ws[i - k] : 0.0;
      double acc = 0.0;
#pragma unroll 4
      for (int t = lane; t < len; t += 32) {
        double y = row[t];
        if (k > 0) {
          y = fma(-wi, v[t + 1], fma(-vi, ws[t + 1], y));
          row[t] = y;
        }
        if (i == k + 1) rbuf[t] = y;
        acc = fma(y, vn[t], acc);
      }
      acc = warp_sum(acc);
      if (lane == 0) pbuf[i - k - 1] = bk * acc;
    }
    grid_barrier(bar, status, G);
    double* sw = v;
    v = vn;
    vn = sw;
    double p[TDG_PER], pv = 0.0;
    const double p0 = __ldcg(pbuf);
#pragma unroll
    for (int j = 0; j < TDG_PER; ++j) {
      const int t = tid + TDG_THREADS * j;
      p[j] = t < len ? __ldcg(pbuf + t) : 0.0;
      x[j] = t < len ? __ldcg(rbuf + t) : 0.0;
    }
#pragma unroll
    for (int j = 0; j < TDG_PER; ++j) {
      const int t = tid + TDG_THREADS * j;
      if (t < len) pv = fma(p[j], v[t], pv);
    }
    pv = partial_sum(pv, len);
    if (tid == 0) sc[0] = 0.5 * bk * pv;
    __syncthreads();
    const double Kc = sc[0], v0 = v[0], w0 = fma(-Kc, v0, p0);
#pragma unroll
    for (int j = 0; j < TDG_PER; ++j) {
      const int t = tid + TDG_THREADS * j;
      if (t < len) {
        const double vt = v[t], wt = fma(-Kc, vt, p[j]);
        ws[t] = wt;
        x[j] = fma(-w0, vt, fma(-v0, wt, x[j]));   // the update of row k + 1, as its owner forms it
      }
    }
    if (k + 3 < n) reflect(k + 1);
  }
  // the last two rows: row n - 2 in x; the last diagonal entry from its owner
  __syncthreads();
  if (rank == 0 && tid < 2) {
    (tid == 0 ? d : e)[n - 2] = x[0];
    beta[n - 2 + tid] = 0.0;
    if (tid == 1) e[n - 1] = 0.0;
  }
  if ((n - 1) % G == rank && tid == 0)
    d[n - 1] = fma(-ws[1], v[1], fma(-v[1], ws[1], rows[(size_t)((n - 1) / G) * n + n - 1]));
}

// ---------------------------------------------------------------------------------
// Eigenvalues of the symmetric tridiagonal T (diagonal d, off-diagonal e) by Sturm-count
// multisection: warp k finds the k-th smallest eigenvalue.  Each lane counts the
// eigenvalues below one of 32 interior points of the current interval (Sturm count);
// the first point whose count exceeds k bounds the eigenvalue from above, its left
// neighbour from below, so each round shrinks the interval 33x.  The start interval is
// Gershgorin's; it is refined to a width of 4 eps ||T|| (what Sturm counts resolve),
// about 11 rounds, or until rounding stops it shrinking.
// ---------------------------------------------------------------------------------
// Number of eigenvalues of T below x: the negative pivots of T - x I,
// q_i = (d_i - x) - e_{i-1}^2 / q_{i-1}; a pivot smaller than pivmin counts as -pivmin.  d and
// e^2 in shared memory; signs and magnitudes by integer compares of the bits (an FP64 compare
// holds the pipe like an FMA: with the squares 8 of them a step, 5 now).
__device__ __forceinline__ int fd_sturm_count(const double* d, const double* e2, int n, double x, double pivmin) {
  const long long pbits = __double_as_longlong(pivmin);
  int cnt = 0;
  double q = d[0] - x;
  auto fix = [&] {
    const long long mag = __double_as_longlong(q) & 0x7fffffffffffffffll;
    if (mag < pbits) q = -pivmin;
    cnt += (__double2hiint(q) < 0 && mag <= 0x7ff0000000000000ll) ? 1 : 0;
  };
  fix();
#pragma unroll 4
  for (int i = 1; i < n; ++i) {
    q = (d[i] - x) - e2[i - 1] * taps_rcp(q);
    fix();
  }
  return cnt;
}

__global__ void fd_bisect_kernel(const double* __restrict__ d, const double* __restrict__ e, int n,
                                 double* __restrict__ lam) {
  extern __shared__ double bs[];   // d [n], e^2 [n]
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    bs[i] = d[i];
    bs[n + i] = e[i] * e[i];
  }
  __syncthreads();
  const int k = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (k >= n) return;   // whole warps
  double lo = INFINITY, hi = -INFINITY, e2max = 0.0;
  for (int i = lane; i < n; i += 32) {
    const double r = (i > 0 ? fabs(e[i - 1]) : 0.0) + (i < n - 1 ? fabs(e[i]) : 0.0);
    lo = fmin(lo, d[i] - r);
    hi = fmax(hi, d[i] + r);
    if (i < n - 1) e2max = fmax(e2max, e[i] * e[i]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    e2max = fmax(e2max, __shfl_xor_sync(0xffffffffu, e2max, o));
  }
  const double eps = 2.220446049250313e-16;
  const double tnorm = fmax(fabs(lo), fabs(hi));
  // underflow guard for the Sturm pivots (the smallest normal double times the largest
  // squared off-diagonal), small enough not to limit the eigenvalues' accuracy
  const double pivmin = 2.2250738585072014e-308 * fmax(1.0, e2max);
  lo -= 4.0 * eps * tnorm + pivmin;
  hi += 4.0 * eps * tnorm + pivmin;
  double wprev = INFINITY;
  for (int it = 0; it < 40; ++it) {
    const double w = hi - lo;
    // Sturm counts resolve an eigenvalue to about eps ||T|| (absolute)
    if (w <= 4.0 * eps * tnorm + pivmin) break;
    if (it > 0 && !(w < wprev)) break;   // rounding no longer separates the trial points
    wprev = w;
    const double x = lo + w * (double)(lane + 1) / 33.0;
    const unsigned above = __ballot_sync(0xffffffffu, fd_sturm_count(bs, bs + n, n, x, pivmin) > k);
    const int j = above ? __ffs(above) - 1 : 32;
    const double nhi = (j < 32) ? lo + w * (double)(j + 1) / 33.0 : hi;
    const double nlo = (j > 0) ? lo + w * (double)j / 33.0 : lo;
    lo = nlo;
    hi = nhi;
  }
  if (lane == 0) lam[k] = 0.5 * (lo + hi);
}

// ---------------------------------------------------------------------------------
// Eigenvectors of T by inverse iteration: thread k factors T - lam_k I by Gaussian
// elimination with partial pivoting (U has two super-diagonals) and solves three times
// from a fixed start vector, normalising after each solve.  Eigenvalues closer than
// FD_CLUSTER ||T|| form a cluster, handled in order by the thread of its first member, each
// iterate orthogonalised against the members already done (modified Gram-Schmidt).  Vectors
// iterated independently are orthogonal to a few eps ||T|| / gap (1.8e-11 at a gap of
// 3e-7 ||T||), which the orthogonalisation step below squares, so the limit lies where that is
// far under eps; the ends of a stiffness pencil's spectrum have gaps of ~2 / n^2 ||T||, and a
// limit of 1e-5 ||T|| made serial clusters of them from 500 nodes on (1532 nodes:
// 95 ms, 11.5 ms now).
// Z is n x n row-major (column k = eigenvector k); W holds five n x n arrays laid out
// [array][row][k] so that neighbouring threads touch neighbouring words.
// ---------------------------------------------------------------------------------
#define FD_CLUSTER 3e-7
__global__ void fd_invit_kernel(const double* __restrict__ d, const double* __restrict__ e,
                                const double* __restrict__ lam, int n, double* __restrict__ Z,
                                double* __restrict__ W) {
  const int k0 = blockIdx.x * blockDim.x + threadIdx.x;
  if (k0 >= n) return;
  double tnorm = 0.0;   // Gershgorin bound of ||T||
  for (int i = 0; i < n; ++i)
    tnorm = fmax(tnorm, fabs(d[i]) + (i > 0 ? fabs(e[i - 1]) : 0.0) + (i + 1 < n ? fabs(e[i]) : 0.0));
  if (!(tnorm > 0.0)) tnorm = 1.0;
  const double ctol = FD_CLUSTER * tnorm;
  if (k0 > 0 && lam[k0] - lam[k0 - 1] <= ctol) return;   // not the first member of its cluster
  int k1 = k0;
  while (k1 + 1 < n && lam[k1 + 1] - lam[k1] <= ctol) ++k1;
  const double tiny = 2.220446049250313e-16 * tnorm;
  const size_t nn = (size_t)n * n;
#define WA(a, i) W[(size_t)(a) * nn + (size_t)(i) * n + k]
#define ZC(i) Z[(size_t)(i) * n + k]
  for (int k = k0; k <= k1; ++k) {
    const double lk = lam[k];
    // ---- factor T - lk I: arrays 0: 1/U0, 1: U1, 2: U2, 3: multiplier, 4: row swap
    double ai = d[0] - lk, bi = n > 1 ? e[0] : 0.0;
    for (int i = 0; i + 1 < n; ++i) {
      const double ci = e[i], an = d[i + 1] - lk, bn = (i + 2 < n) ? e[i + 1] : 0.0;
      if (fabs(ai) >= fabs(ci)) {
        if (ai == 0.0) ai = tiny;
        const double m = ci / ai;
        WA(0, i) = 1.0 / ai;
        WA(1, i) = bi;
        WA(2, i) = 0.0;
        WA(3, i) = m;
        WA(4, i) = 0.0;
        ai = an - m * bi;
        bi = bn;
      } else {
        const double m = ai / ci;
        WA(0, i) = 1.0 / ci;
        WA(1, i) = an;
        WA(2, i) = bn;
        WA(3, i) = m;
        WA(4, i) = 1.0;
        ai = bi - m * an;
        bi = -m * bn;
      }
    }
    if (ai == 0.0) ai = tiny;
    WA(0, n - 1) = 1.0 / ai;
    WA(1, n - 1) = 0.0;   // the last row has no super-diagonals
    WA(2, n - 1) = 0.0;
    // ---- start vector (fixed, different per k), then three solves
    for (int i = 0; i < n; ++i) ZC(i) = 1.0 + 0.5 * sin(0.7 * i + 1.3 * k);
    for (int it = 0; it < 3; ++it) {
      // forward: row swaps and multipliers (the running entry stays in a register)
      double yi = ZC(0);
#pragma unroll 8
      for (int i = 0; i + 1 < n; ++i) {
        double yn = ZC(i + 1);
        if (WA(4, i) != 0.0) {
          const double t = yi;
          yi = yn;
          yn = t;
        }
        ZC(i) = yi;
        yi = yn - WA(3, i) * yi;
      }
      ZC(n - 1) = yi;
      // backward with the two super-diagonals (z_{i+1}, z_{i+2} in registers)
      double z1 = 0.0, z2 = 0.0;
#pragma unroll 8
      for (int i = n - 1; i >= 0; --i) {
        const double zi = (ZC(i) - WA(1, i) * z1 - WA(2, i) * z2) * WA(0, i);
        ZC(i) = zi;
        z2 = z1;
        z1 = zi;
      }
      for (int j = k0; j < k; ++j) {   // against the cluster's earlier members
        double dot = 0.0;
        for (int i = 0; i < n; ++i) dot += Z[(size_t)i * n + j] * ZC(i);
        for (int i = 0; i < n; ++i) ZC(i) -= dot * Z[(size_t)i * n + j];
      }
      double nrm = 0.0;
      for (int i = 0; i < n; ++i) nrm += ZC(i) * ZC(i);
      const double inv = (nrm > 0.0) ? 1.0 / sqrt(nrm) : 0.0;
      for (int i = 0; i < n; ++i) ZC(i) *= inv;
    }
  }
#undef WA
#undef ZC
}

// The same with T, the factors and the iterate in shared memory: IV_COLS eigenvectors to a CTA
// of one warp, as many of 8, 4, 2, 1 as fit (n <= ~820, 1560, 2820, 4720).  The passes are chains
// over the nodes whose global-memory arrays, written and read back by the same thread, were most
// of their time (254 nodes: 1055 and 644 us; 1532 nodes, 4 to a CTA: 157 and 95 ms, 11.5 with the
// narrower clusters).
static size_t iv_smem(int n, int cols) {
  return sizeof(double) * (2 * (size_t)n + 4 * (size_t)n * cols) + (size_t)n * cols;
}

template <int IV_COLS>
__global__ void __launch_bounds__(32) fd_invit_smem_kernel(const double* __restrict__ dg, const double* __restrict__ eg,
                                                           const double* __restrict__ lam, int n,
                                                           double* __restrict__ Z) {
  extern __shared__ double ism[];
  double* d = ism;
  double* e = ism + n;
  double* W = ism + 2 * n;                         // [3][n][IV_COLS]: 1/U0, U1, multiplier
  double* z = W + 3 * (size_t)n * IV_COLS;         // [n][IV_COLS]
  unsigned char* swap = reinterpret_cast<unsigned char*>(z + (size_t)n * IV_COLS);
  const int l = threadIdx.x;
  for (int i = l; i < n; i += 32) {
    d[i] = dg[i];
    e[i] = eg[i];
  }
  __syncwarp();
  const int k0 = blockIdx.x * IV_COLS + l;
  if (l >= IV_COLS || k0 >= n) return;
  double tnorm = 0.0;   // Gershgorin bound of ||T||
  for (int i = 0; i < n; ++i)
    tnorm = fmax(tnorm, fabs(d[i]) + (i > 0 ? fabs(e[i - 1]) : 0.0) + (i + 1 < n ? fabs(e[i]) : 0.0));
  if (!(tnorm > 0.0)) tnorm = 1.0;
  const double ctol = FD_CLUSTER * tnorm;
  if (k0 > 0 && lam[k0] - lam[k0 - 1] <= ctol) return;   // not the first member of its cluster
  int k1 = k0;
  while (k1 + 1 < n && lam[k1 + 1] - lam[k1] <= ctol) ++k1;
  const double tiny = 2.220446049250313e-16 * tnorm;
#define WA(a, i) W[((size_t)(a) * n + (i)) * IV_COLS + l]
#define SW(i) swap[(size_t)(i) * IV_COLS + l]
#define ZC(i) z[(size_t)(i) * IV_COLS + l]
  for (int k = k0; k <= k1; ++k) {
    const double lk = lam[k];
    double ai = d[0] - lk, bi = n > 1 ? e[0] : 0.0;
    for (int i = 0; i + 1 < n; ++i) {
      const double ci = e[i], an = d[i + 1] - lk, bn = (i + 2 < n) ? e[i + 1] : 0.0;
      // both sides of the pivoting in one: its two divisions (a dozen FP64 instructions each)
      // are not issued for either side
      const bool keep = fabs(ai) >= fabs(ci);
      if (keep && ai == 0.0) ai = tiny;
      const double den = keep ? ai : ci, num = keep ? ci : ai;
      const double m = num / den;
      WA(0, i) = 1.0 / den;
      WA(1, i) = keep ? bi : an;
      WA(2, i) = m;
      SW(i) = keep ? 0 : 1;
      const double upper = keep ? bi : an;
      ai = (keep ? an : bi) - m * upper;
      bi = keep ? bn : -m * bn;
    }
    if (ai == 0.0) ai = tiny;
    WA(0, n - 1) = 1.0 / ai;
    WA(1, n - 1) = 0.0;   // the last row has no super-diagonals
    SW(n - 1) = 0;
    for (int i = 0; i < n; ++i) ZC(i) = 1.0 + 0.5 * sin(0.7 * i + 1.3 * k);
    for (int it = 0; it < 3; ++it) {
      double yi = ZC(0);
#pragma unroll 4
      for (int i = 0; i + 1 < n; ++i) {
        double yn = ZC(i + 1);
        if (SW(i)) {
          const double t = yi;
          yi = yn;
          yn = t;
        }
        ZC(i) = yi;
        yi = yn - WA(2, i) * yi;
      }
      ZC(n - 1) = yi;
      double z1 = 0.0, z2 = 0.0;
#pragma unroll 4
      for (int i = n - 1; i >= 0; --i) {
        const double u2 = SW(i) && i + 2 < n ? e[i + 1] : 0.0;   // filled in by an exchange of rows
        const double zi = (ZC(i) - WA(1, i) * z1 - u2 * z2) * WA(0, i);
        ZC(i) = zi;
        z2 = z1;
        z1 = zi;
      }
      for (int j = k0; j < k; ++j) {   // against the cluster's earlier members
        double dot = 0.0;
        for (int i = 0; i < n; ++i) dot += Z[(size_t)i * n + j] * ZC(i);
        for (int i = 0; i < n; ++i) ZC(i) -= dot * Z[(size_t)i * n + j];
      }
      double nrm = 0.0;
#pragma unroll 4
      for (int i = 0; i < n; ++i) nrm += ZC(i) * ZC(i);
      const double inv = (nrm > 0.0) ? 1.0 / sqrt(nrm) : 0.0;
      for (int i = 0; i < n; ++i) ZC(i) *= inv;
    }
    for (int i = 0; i < n; ++i) Z[(size_t)i * n + k] = ZC(i);
  }
#undef WA
#undef SW
#undef ZC
}

// ---------------------------------------------------------------------------------
// Symmetric orthogonalisation of the inverse-iteration vectors, first order:
// Z <- Z - Z E / 2 with E = Z^T Z - I.  Independently computed eigenvectors are
// orthogonal only to ~eps ||T|| / gap (1e-11 for the lowest eigenvalues of a stiffness
// pencil); one step squares that, and Z^T T Z stays diagonal to ~eps ||T|| because the
// correction of entry (j, k) is scaled by lam_j + lam_k.  E[j][k]: one thread each;
// four partial sums shorten the dependent FP64 chain.
// ---------------------------------------------------------------------------------
__global__ void fd_gram_minus_identity_kernel(const double* __restrict__ Z, int n, double* __restrict__ E) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)n * n) return;
  const int j = (int)(idx / n), k = (int)(idx % n);
  double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
  int i = 0;
  for (; i + 3 < n; i += 4) {
    a0 += Z[(size_t)i * n + j] * Z[(size_t)i * n + k];
    a1 += Z[(size_t)(i + 1) * n + j] * Z[(size_t)(i + 1) * n + k];
    a2 += Z[(size_t)(i + 2) * n + j] * Z[(size_t)(i + 2) * n + k];
    a3 += Z[(size_t)(i + 3) * n + j] * Z[(size_t)(i + 3) * n + k];
  }
  for (; i < n; ++i) a0 += Z[(size_t)i * n + j] * Z[(size_t)i * n + k];
  E[idx] = ((a0 + a1) + (a2 + a3)) - (j == k ? 1.0 : 0.0);
}

__global__ void fd_orth_update_kernel(const double* __restrict__ Z, const double* __restrict__ E, int n,
                                      double* __restrict__ Zout) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)n * n) return;
  const int i = (int)(idx / n), k = (int)(idx % n);
  const double* zi = Z + (size_t)i * n;
  double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
  int j = 0;
  for (; j + 3 < n; j += 4) {
    a0 += zi[j] * E[(size_t)j * n + k];
    a1 += zi[j + 1] * E[(size_t)(j + 1) * n + k];
    a2 += zi[j + 2] * E[(size_t)(j + 2) * n + k];
    a3 += zi[j + 3] * E[(size_t)(j + 3) * n + k];
  }
  for (; j < n; ++j) a0 += zi[j] * E[(size_t)j * n + k];
  Zout[idx] = zi[k] - 0.5 * ((a0 + a1) + (a2 + a3));
}

// ---------------------------------------------------------------------------------
// Back-transform Z <- Q Z with Q = H_0 H_1 ... H_{n-3}, H_r = I - beta_r v_r v_r^T acting
// on rows r+1 .. n-1 (v_r in row r of V): warp c takes column c through the reflections
// from the last to the first, the column held in shared memory.
// ---------------------------------------------------------------------------------
#define BT_REGS 16   // reflector entries per lane held in registers (n <= 512)
__global__ void fd_backtransform_kernel(const double* __restrict__ V, const double* __restrict__ beta, int n,
                                        double* __restrict__ Z) {
  extern __shared__ double zs[];   // [warps per CTA][n]
  const int wl = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c = blockIdx.x * (blockDim.x >> 5) + wl;
  if (c >= n) return;   // whole warps
  double* z = zs + (size_t)wl * n;
  for (int i = lane; i < n; i += 32) z[i] = Z[(size_t)i * n + c];
  __syncwarp();
  if (n <= 32 * BT_REGS) {
    // the next reflector is loaded while one is applied
    double v[BT_REGS], nv[BT_REGS], br = 0.0, nbr = 0.0;
    auto load = [&](int r) {
      if (r < 0) return;
      nbr = beta[r];
#pragma unroll
      for (int t = 0; t < BT_REGS; ++t) {
        const int i = r + 1 + lane + 32 * t;
        nv[t] = i < n ? V[(size_t)r * n + i] : 0.0;
      }
    };
    load(n - 3);
    for (int r = n - 3; r >= 0; --r) {
      br = nbr;
#pragma unroll
      for (int t = 0; t < BT_REGS; ++t) v[t] = nv[t];
      load(r - 1);
      if (br == 0.0) continue;
      double dot = 0.0;
#pragma unroll
      for (int t = 0; t < BT_REGS; ++t) {
        const int i = r + 1 + lane + 32 * t;
        if (r + 1 + 32 * t >= n) break;   // the same for every lane
        if (i < n) dot += v[t] * z[i];
      }
      dot = warp_sum(dot) * br;
#pragma unroll
      for (int t = 0; t < BT_REGS; ++t) {
        const int i = r + 1 + lane + 32 * t;
        if (r + 1 + 32 * t >= n) break;
        if (i < n) z[i] -= dot * v[t];
      }
      __syncwarp();
    }
  } else {
    for (int r = n - 3; r >= 0; --r) {
      const double br = beta[r];
      if (br == 0.0) continue;
      const double* v = V + (size_t)r * n;
      double dot = 0.0;
      for (int i = r + 1 + lane; i < n; i += 32) dot += v[i] * z[i];
      dot = warp_sum(dot) * br;
      for (int i = r + 1 + lane; i < n; i += 32) z[i] -= dot * v[i];
      __syncwarp();
    }
  }
  for (int i = lane; i < n; i += 32) Z[(size_t)i * n + c] = z[i];
}

// Phi = L^{-T} Z (L: the banded Cholesky factor in B, lower, half-width hb), Phi^T, and
// mu = the eigenvalues; one thread per column.  Without an A (single-operator pencil)
// Z = I and mu = 0.
template <int HB>
__global__ void __launch_bounds__(32) fd_phi_kernel(const double* __restrict__ L, const double* __restrict__ linv,
                                                    const double* __restrict__ Z, const double* __restrict__ lam, int n,
                                                    double* __restrict__ Phi, double* __restrict__ PhiT,
                                                    double* __restrict__ mu, int* status) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n) return;
  double x[HB];                                   // values of rows i + 1 .. i + HB
  double l[FD_AHEAD][HB], in[FD_AHEAD], li[FD_AHEAD];
  auto load = [&](int i, double (&p)[HB], double& q, double& r) {
    if (i < 0) return;
#pragma unroll
    for (int t = 0; t < HB; ++t) p[t] = i + 1 + t < n ? L[(size_t)(i + 1 + t) * n + i] : 0.0;
    q = Z ? Z[(size_t)i * n + c] : (i == c ? 1.0 : 0.0);
    r = linv[i];
  };
#pragma unroll
  for (int t = 0; t < HB; ++t) x[t] = 0.0;
#pragma unroll
  for (int a = 0; a < FD_AHEAD; ++a) load(n - 1 - a, l[a], in[a], li[a]);
  for (int i0 = n - 1; i0 >= 0; i0 -= FD_AHEAD) {
#pragma unroll
    for (int a = 0; a < FD_AHEAD; ++a) {
      const int i = i0 - a;
      if (i < 0) break;
      double s = in[a];
#pragma unroll
      for (int t = 0; t < HB; ++t)
        if (i + 1 + t < n) s -= l[a][t] * x[t];
      s = s * li[a];
      Phi[(size_t)i * n + c] = s;
      PhiT[(size_t)c * n + i] = s;
#pragma unroll
      for (int t = HB - 1; t > 0; --t) x[t] = x[t - 1];
      x[0] = s;
      load(i - FD_AHEAD, l[a], in[a], li[a]);
    }
  }
  const double m = lam ? lam[c] : 0.0;
  mu[c] = m;
  if (!isfinite(m)) taps_flag(status, TAPS_DEV_NONFINITE);
}

// ---------------------------------------------------------------------------------
// Per-solve kernels
// ---------------------------------------------------------------------------------
// F[i][m] = sum_r q_r[i] c_r[m], one FMA chain per entry.
__global__ void __launch_bounds__(128) fd_rhs_kernel(const double* __restrict__ q, const double* __restrict__ c,
                                                     int Rf, int nf, int M, double* __restrict__ F) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)nf * M) return;
  const int i = (int)(idx / M), m = (int)(idx % M);
  F[idx] = taps_fma_chain<16>(
      Rf, [&](int r) { return q[(size_t)r * nf + i]; }, [&](int r) { return c[(size_t)r * M + m]; });
}

// The same with the sum over r in four parts, one per warp of a CTA of 32 entries.
__global__ void __launch_bounds__(128) fd_rhs_split_kernel(const double* __restrict__ q, const double* __restrict__ c,
                                                           int Rf, int nf, int M, double* __restrict__ F) {
  __shared__ double part[4][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long idx = (long long)blockIdx.x * 32 + lane;
  const bool in = idx < (long long)nf * M;
  const int i = in ? (int)(idx / M) : 0, m = in ? (int)(idx % M) : 0;
  const int r0 = Rf * w / 4, r1 = Rf * (w + 1) / 4;
  const double *qi = q + (size_t)r0 * nf + i, *cm = c + (size_t)r0 * M + m;
  part[w][lane] = taps_fma_chain<16>(
      r1 - r0, [&](int r) { return qi[(size_t)r * nf]; }, [&](int r) { return cm[(size_t)r * M]; });
  __syncthreads();
  if (w == 0 && in) F[idx] = (part[0][lane] + part[1][lane]) + (part[2][lane] + part[3][lane]);
}

// The chain of R_f dependent FMAs bounds a moving source's hundreds of terms while the entries
// leave most sub-partitions idle; beyond a warp per sub-partition the FP64 issue does, and
// splitting the chain gives nothing.  466 terms, 255 nodes of 20 modes: 47 us as one
// chain, 16 us in four; 239 terms, 1534 nodes of 100 modes: 95 us as one chain.
int taps_rhs(const double* q, const double* c, int Rf, int n, int M, double* F, int num_sms, cudaStream_t s) {
  const long long nM = (long long)n * M;
  if (Rf >= 128 && nM <= 128ll * num_sms)
    fd_rhs_split_kernel<<<(unsigned)((nM + 31) / 32), 128, 0, s>>>(q, c, Rf, n, M, F);
  else
    fd_rhs_kernel<<<(unsigned)((nM + 127) / 128), 128, 0, s>>>(q, c, Rf, n, M, F);
  TAPS_CUDA(cudaGetLastError());
  return TAPS_OK;
}

// PQ[r][i] = sum_j PhiT[i][j] q[r][j]: the source vectors of dim d in the eigenbasis
// of its pencil.  The reduced right-hand side of dim d is F = Q c (c from the other
// dims), so its transform Phi^T F = (Phi^T Q) c needs only this fixed n x Rf matrix.
// (Read through Phi, whose neighbouring threads' entries are neighbours.)
__global__ void __launch_bounds__(128) fd_pq_kernel(const double* __restrict__ Phi, const double* __restrict__ q, int n,
                                                    int Rf, double* __restrict__ PQ) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)n * Rf) return;
  const int r = (int)(idx / n), i = (int)(idx % n);
  const double* qr = q + (size_t)r * n;
  PQ[idx] = taps_fma_chain<16>(n, [&](int j) { return Phi[(size_t)j * n + i]; }, [&](int j) { return qr[j]; });
}

// Out[i][m] = sum_j Mat[i][j] In[j][m] (Mat n x n row-major, In n x M row-major).
// One CTA per output row i.  Its RG_WARPS warps (one per SM sub-partition) split the
// sum over j; within a warp the lanes split it again, each lane keeping 32 mode
// accumulators.  A butterfly reduce-scatter then leaves lane l of each warp with the
// warp's sum for mode l (31 additions per lane instead of a chain of 32), and the
// warps' sums are combined through shared memory.  FP64 on this GPU is issue-bound
// per sub-partition, so spreading one row over all four pipes matters.
// Out is n x M row-major, or (colmajor) the factor layout Out[m * n + i]; in the
// factor layout a non-null Save receives the row's previous values first.
#define RG_WARPS 4
__global__ void __launch_bounds__(RG_WARPS * 32) fd_rowgemm_kernel(const double* __restrict__ Mat,
                                                                   const double* __restrict__ In, int n,
                                                                   int M, double* __restrict__ Out,
                                                                   int colmajor,
                                                                   double* __restrict__ Save) {
  __shared__ double part[RG_WARPS][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x;
  taps_pdl_wait();
  if (colmajor && Save)   // the writes below come after a barrier
    for (int m = threadIdx.x; m < M; m += blockDim.x) Save[(size_t)m * n + i] = Out[(size_t)m * n + i];
  const double* row = Mat + (size_t)i * n;
  const int step = RG_WARPS * 32;
  for (int m0 = 0; m0 < M; m0 += 32) {
    const int mc = min(32, M - m0);
    double acc[32];
#pragma unroll
    for (int c = 0; c < 32; ++c) acc[c] = 0.0;
    for (int j = warp * 32 + lane; j < n; j += step) {
      const double a = row[j];
      const double* in = In + (size_t)j * M + m0;
#pragma unroll
      for (int c = 0; c < 32; ++c)
        if (c < mc) acc[c] += a * in[c];
    }
    // reduce-scatter: at offset o a lane keeps the half of its current modes selected
    // by lane bit o and receives its partner's values of that half
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int c = 0; c < o; ++c) {
        const double send = up ? acc[c] : acc[c + o];
        const double keep = up ? acc[c + o] : acc[c];
        acc[c] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
    }
    part[warp][lane] = acc[0];   // the warp's sum for mode m0 + lane
    __syncthreads();
    if (threadIdx.x < mc) {
      const double sum = (part[0][threadIdx.x] + part[1][threadIdx.x]) +
                         (part[2][threadIdx.x] + part[3][threadIdx.x]);
      if (colmajor) Out[(size_t)(m0 + threadIdx.x) * n + i] = sum;
      else Out[(size_t)i * M + m0 + threadIdx.x] = sum;
    }
    __syncthreads();
  }
}

// The same product as a tiled contraction for many rows and modes: a CTA takes 32 rows (lane =
// row) of four modes (warp = mode, so that a mode count that is no multiple of the tile wastes
// no FP64 issue), 32 columns of Mat at a time through two shared buffers, the next ones loaded
// while these are multiplied.  Each tile is four chains of 8, and the tiles are added in pairs up
// to eight, so that an entry's rounding stays that of the row kernel's short sums (6.9e-15 against
// 6.8e-15 rms over 1534 normal products).  The row kernel pays a butterfly
// per row and 32 modes and an L1 line per lane and operand; FP64 issue is the bound of this one.
// 1534 rows of 100 modes: 621 us with a CTA per row, 461 us.
#define FM_TILE 32
#define FM_WARPS 4
__global__ void __launch_bounds__(FM_WARPS * 32) fd_matmul_kernel(const double* __restrict__ Mat,
                                                                  const double* __restrict__ In, int n, int M,
                                                                  double* __restrict__ Out, int colmajor,
                                                                  double* __restrict__ Save) {
  __shared__ double As[2][FM_TILE][FM_TILE + 1];   // [column of Mat][row]
  __shared__ double Bs[2][FM_TILE][FM_WARPS];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int i0 = blockIdx.x * FM_TILE, m0 = blockIdx.y * FM_WARPS;
  const int i = i0 + lane, m = m0 + warp;
  double ra[FM_TILE / FM_WARPS], rb;
  auto load = [&](int k0) {
    const int k = k0 + lane;
#pragma unroll
    for (int e = 0; e < FM_TILE / FM_WARPS; ++e) {
      const int r = i0 + warp + FM_WARPS * e;
      ra[e] = (r < n && k < n) ? Mat[(size_t)r * n + k] : 0.0;
    }
    const int kb = k0 + tid / FM_WARPS, mb = m0 + tid % FM_WARPS;
    rb = (kb < n && mb < M) ? In[(size_t)kb * M + mb] : 0.0;
  };
  taps_pdl_wait();
  load(0);
  double sum = 0.0, one = 0.0, two = 0.0, four = 0.0;
  int t = 0;
  for (int k0 = 0; k0 < n; k0 += FM_TILE, ++t) {
    const int cur = t & 1;
#pragma unroll
    for (int e = 0; e < FM_TILE / FM_WARPS; ++e) As[cur][lane][warp + FM_WARPS * e] = ra[e];
    Bs[cur][tid / FM_WARPS][tid % FM_WARPS] = rb;
    __syncthreads();   // the other buffer's readers are past it as well
    if (k0 + FM_TILE < n) load(k0 + FM_TILE);
    if (m < M) {
      double a[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
      for (int k = 0; k < FM_TILE / 4; ++k)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int kc = k + c * (FM_TILE / 4);
          a[c] = fma(As[cur][kc][lane], Bs[cur][kc][warp], a[c]);
        }
      double x = (a[0] + a[1]) + (a[2] + a[3]);
      // pairwise up to eight tiles
      if (!(t & 1)) one = x;
      else {
        x += one;
        if (!(t & 2)) two = x;
        else {
          x += two;
          if (!(t & 4)) four = x;
          else sum += x + four;
        }
      }
    }
  }
  if (m >= M || i >= n) return;
  if (t & 4) sum += four;
  if (t & 2) sum += two;
  if (t & 1) sum += one;
  if (!colmajor) {
    Out[(size_t)i * M + m] = sum;
    return;
  }
  double* o = Out + (size_t)m * n + i;
  if (Save) Save[(size_t)m * n + i] = *o;
  *o = sum;
}

// The tiled product beyond 32 modes, where the row kernel takes more than one pass over Mat and
// its lanes' operands lie further apart (64 modes: 9.6 and 5.0 us for 12 rows, 25 and 17 for 254,
// 46 and 34 for 382, 87 and 51 for 606; 40 modes: 191 and 140 us for 1214 rows).  Up to 32 modes
// its tiles are too few and their chains the longer ones (254 rows of 30 modes: 10.6 and 16.8 us).
static int fd_transform(const double* Mat, const double* In, int n, int M, double* Out, int colmajor, double* Save,
                        cudaStream_t s) {
  if (M > 32)
    TAPS_CUDA(taps_launch_pdl(fd_matmul_kernel, dim3((n + FM_TILE - 1) / FM_TILE, (M + FM_WARPS - 1) / FM_WARPS),
                              dim3(FM_WARPS * 32), 0, s, Mat, In, n, M, Out, colmajor, Save));
  else
    TAPS_CUDA(taps_launch_pdl(fd_rowgemm_kernel, dim3(n), dim3(RG_WARPS * 32), 0, s, Mat, In, n, M, Out, colmajor,
                              Save));
  return TAPS_OK;
}

// One warp per node i, M <= 32: lane r holds row r of (mu_i C_A + C_B | g_i) in
// registers.  Without refinement: LU without pivoting in FP64 (the systems have a
// positive definite symmetric part) and back substitution by shuffles.  With
// refinement: the LU runs in FP32 (whose dependent-instruction latency is a small
// fraction of FP64's on this GPU) and the solution is refined in FP64
// (y += T^{-1}_32 (g - T y)) until the FP64 residual is at the level of FP64
// rounding; a system that does not get there in 4 steps is solved again by the FP64
// LU.  A zero or non-finite pivot is reported as TAPS_DEV_SINGULAR.
template <typename R>
__device__ __forceinline__ void warp_lu_inplace(R row[33], int lane, int M, bool& bad) {
#pragma unroll
  for (int p = 0; p < 32; ++p) {
    if (p < M) {
      R piv = __shfl_sync(0xffffffffu, row[p], p);
      bad |= !(fabs((double)piv) > 0.0) || !isfinite((double)piv);
      R l = (lane > p && lane < M && piv != (R)0) ? row[p] / piv : (R)0;
#pragma unroll
      for (int c = 0; c < 32; ++c) {
        if (c > p && c < M) {
          R pc = __shfl_sync(0xffffffffu, row[c], p);
          row[c] -= l * pc;
        }
      }
      if (lane > p && lane < M) row[p] = l;   // keep the multiplier (unit lower L)
    }
  }
}

// Solve L U x = b with the factors of warp_lu_inplace; b and x are lane-distributed.
template <typename R>
__device__ __forceinline__ R warp_lu_solve(const R row[33], R b, int lane, int M) {
#pragma unroll
  for (int p = 0; p < 32; ++p) {
    if (p < M) {
      R bp = __shfl_sync(0xffffffffu, b, p);
      if (lane > p && lane < M) b -= row[p] * bp;
    }
  }
  R x = (R)0;
#pragma unroll
  for (int c = 31; c >= 0; --c) {
    if (c < M) {
      R xc = (lane == c && row[c] != (R)0) ? b / row[c] : (R)0;
      xc = __shfl_sync(0xffffffffu, xc, c);
      if (lane == c) x = xc;
      if (lane < c) b -= row[c] * xc;
    }
  }
  return x;
}

__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

__global__ void __launch_bounds__(32) fd_small_solve_warp_kernel(const double* __restrict__ CA,
                                                                 const double* __restrict__ CB,
                                                                 const double* __restrict__ mu,
                                                                 const double* __restrict__ G, int n,
                                                                 int M, double* __restrict__ Y,
                                                                 int* status, int refine) {
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.x;   // one warp per CTA: the n systems spread over every SM
  if (i >= n) return;
  const double mi = (CA && mu) ? mu[i] : 0.0;
  double row[33];
#pragma unroll
  for (int c = 0; c < 32; ++c) {
    double v = 0.0;
    if (lane < M && c < M) v = (CA ? mi * CA[lane * M + c] : 0.0) + CB[lane * M + c];
    row[c] = v;
  }
  const double g = (lane < M) ? G[(size_t)i * M + lane] : 0.0;
  bool bad = false;
  double x = 0.0;
  bool done = false;
  if (refine) {
    float rf[33];
#pragma unroll
    for (int c = 0; c < 33; ++c) rf[c] = (float)row[c];
    bool bad32 = false;
    warp_lu_inplace<float>(rf, lane, M, bad32);
    if (!bad32) {
      double tnorm = 0.0;
#pragma unroll
      for (int c = 0; c < 32; ++c) tnorm += fabs(row[c]);
      tnorm = warp_max(tnorm);
      double r = g;
      for (int it = 0; it < 4 && !done; ++it) {
        x += (double)warp_lu_solve<float>(rf, (float)r, lane, M);
        // r = g - T x in FP64, as four independent partial sums (FP64 latency is long)
        double a0 = g, a1 = 0.0, a2 = 0.0, a3 = 0.0;
#pragma unroll
        for (int c = 0; c < 32; c += 4) {
          double x0 = __shfl_sync(0xffffffffu, x, c), x1 = __shfl_sync(0xffffffffu, x, c + 1);
          double x2 = __shfl_sync(0xffffffffu, x, c + 2), x3 = __shfl_sync(0xffffffffu, x, c + 3);
          if (c < M) a0 -= row[c] * x0;
          if (c + 1 < M) a1 -= row[c + 1] * x1;
          if (c + 2 < M) a2 -= row[c + 2] * x2;
          if (c + 3 < M) a3 -= row[c + 3] * x3;
        }
        r = (lane < M) ? (a0 + a1) + (a2 + a3) : 0.0;
        double rmax = warp_max(fabs(r)), xmax = warp_max(fabs(x)), gmax = warp_max(fabs(g));
        // FP64 backward accuracy (a few eps), so that the refined path gives the
        // FP64 path's factors; the FP64 LU below is the fallback
        done = rmax <= 8.0 * 2.220446049250313e-16 * (tnorm * xmax + gmax);
        if (!isfinite(rmax)) break;
      }
    }
  }
  if (!done) {   // FP64 LU (also the fallback of the refined path)
    warp_lu_inplace<double>(row, lane, M, bad);
    x = warp_lu_solve<double>(row, g, lane, M);
    if (bad && lane == 0) taps_flag(status, TAPS_DEV_SINGULAR);
  }
  if (lane < M) Y[(size_t)i * M + lane] = x;
}

// One CTA of four warps per node i, M <= 32, FP64.  FP64 instructions issue at a
// fraction of a lane per clock per SM sub-partition on this GPU, so the elimination
// of one system is spread over the four sub-partitions: warp w holds the columns
// c = w, w+4, w+8, ... of T = mu_i C_A + C_B (lane r = row r) and warp 0 also the
// right-hand side g_i = sum_r PQ[r][i] c_r, formed here from the transformed source
// vectors (the warps split the sum over r).  At step p every warp updates its
// columns c > p with the multipliers l_r = T[r][p] / T[p][p] of that step, which the
// owner of column p has published in shared memory (one reciprocal of the pivot,
// kept for the back substitution).  The chain of pivots is the bound: the owner of
// column p+1 updates that column first (its row-p value fetched before the barrier),
// takes the pivot's reciprocal (approximate seed + series refinement) and issues its
// other updates while the reciprocal completes.  No pivoting, as in the one-warp
// solve.  The upper factor then goes to shared memory and warp 0 back-substitutes.
__global__ void __launch_bounds__(128) fd_small_solve_quad_kernel(const double* __restrict__ CA,
                                                                  const double* __restrict__ CB,
                                                                  const double* __restrict__ mu,
                                                                  const double* __restrict__ PQ,
                                                                  const double* __restrict__ cf, int Rf,
                                                                  int n, int M, double* __restrict__ Y,
                                                                  int* status) {
  __shared__ double gpart[4][32];
  __shared__ double lbuf[2][32];
  __shared__ double invd[32];
  __shared__ double Ush[32][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int i = blockIdx.x;
  if (i >= n) return;
  taps_pdl_wait();
  const double mi = (CA && mu) ? mu[i] : 0.0;
  double v[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int c = 4 * k + w;
    double x = 0.0;
    if (lane < M && c < M) x = (CA ? mi * CA[lane * M + c] : 0.0) + CB[lane * M + c];
    v[k] = x;
  }
  double gp = 0.0;
  if (lane < M)
    for (int r = w; r < Rf; r += 4) gp += PQ[(size_t)r * n + i] * cf[(size_t)r * M + lane];
  gpart[w][lane] = gp;
  bool bad = false;
  // multipliers of step 0 (column 0 belongs to warp 0)
  if (w == 0) {
    const double piv = __shfl_sync(0xffffffffu, v[0], 0);
    bad |= !taps_finite_nonzero(piv);
    const double inv = taps_rcp(piv);
    lbuf[0][lane] = (lane > 0 && lane < M) ? v[0] * inv : 0.0;
    if (lane == 0) invd[0] = inv;
  }
  // row 0 of column 1, for the owner of the next pivot
  double pc_next = (w == 1) ? __shfl_sync(0xffffffffu, v[0], 0) : 0.0;
  __syncthreads();
  double b = (w == 0) ? (gpart[0][lane] + gpart[1][lane]) + (gpart[2][lane] + gpart[3][lane]) : 0.0;
#pragma unroll
  for (int p = 0; p < 32; ++p) {
    if (p < M) {
      const double l = lbuf[p & 1][lane];
      const int q = p + 1;   // next pivot column, owned by warp q & 3 in slot q >> 2
      if (q < M && w == (q & 3)) {
        // owner of column q: that column (its row p was fetched before the barrier),
        // the pivot's reciprocal, then its other columns in the same block so that
        // their FP64 issue fills the reciprocal's latency, then the next multipliers
        v[q >> 2] -= l * pc_next;
        const double piv = __shfl_sync(0xffffffffu, v[q >> 2], q);
        const double inv = taps_rcp(piv);
#pragma unroll
        for (int k = (q >> 2) + 1; k < 8; ++k) v[k] -= l * __shfl_sync(0xffffffffu, v[k], p);
        lbuf[q & 1][lane] = (lane > q && lane < M) ? v[q >> 2] * inv : 0.0;
        if (lane == 0) invd[q] = inv;
        bad |= !taps_finite_nonzero(piv);
      } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) {   // this warp's columns c > p
          if (4 * k + 3 <= p) continue;                 // every column of this slot is <= p
          if (4 * k <= p && w <= p - 4 * k) continue;   // column 4k + w <= p
          v[k] -= l * __shfl_sync(0xffffffffu, v[k], p);
        }
      }
      if (w == 0) b -= l * __shfl_sync(0xffffffffu, b, p);
      // row q of column q + 1 is final now: the next owner fetches it before the barrier
      if (q + 1 < M && w == ((q + 1) & 3)) pc_next = __shfl_sync(0xffffffffu, v[(q + 1) >> 2], q);
      __syncthreads();
    }
  }
  // upper factor to shared memory; warp 0 back-substitutes with the kept reciprocals
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int c = 4 * k + w;
    Ush[lane][c] = v[k];
  }
  __syncthreads();
  if (w == 0) {
    double x = 0.0;
#pragma unroll
    for (int c = 31; c >= 0; --c) {
      if (c < M) {
        const double xc = __shfl_sync(0xffffffffu, b, c) * invd[c];
        if (lane == c) x = xc;
        if (lane < c) b -= Ush[lane][c] * xc;
      }
    }
    if (lane < M) Y[(size_t)i * M + lane] = x;
  }
  if (bad && lane == 0) taps_flag(status, TAPS_DEV_SINGULAR);
}

// One CTA per node i (M > 32): solve (mu_i C_A + C_B) y = g_i by LU with partial pivoting in
// shared memory (small_lu.cuh).  A zero or non-finite pivot is reported as
// TAPS_DEV_SINGULAR.  1534 systems of 100 modes: 1.97 ms with the pivot search between two
// barriers of a step, 1.30 ms now (0.85 ms of FP64 issue).  Eleven update warps beside the pivot's
// load the four sub-partitions more evenly than seven (1.35 ms; 183 and 156 us for 16 systems);
// fifteen take 1.31 ms.
#define FS_THREADS 384
__global__ void __launch_bounds__(FS_THREADS, 2) fd_small_solve_kernel(const double* __restrict__ CA,
                                                                       const double* __restrict__ CB,
                                                                       const double* __restrict__ mu,
                                                                       const double* __restrict__ G, int M,
                                                                       double* __restrict__ Y, int* status) {
  extern __shared__ double T[];   // [M][M+1]: matrix | rhs
  __shared__ SmallLu sh;
  const int i = blockIdx.x, tid = threadIdx.x;
  const int ld = M + 1;
  const double mi = mu ? mu[i] : 0.0;
  for (int idx = tid; idx < M * M; idx += FS_THREADS) {
    int r = idx / M, c = idx % M;
    T[r * ld + c] = (CA ? mi * CA[idx] : 0.0) + CB[idx];
  }
  for (int r = tid; r < M; r += FS_THREADS) T[r * ld + M] = G[(size_t)i * M + r];
  double b[TAPS_MAX_M / 32];
  bool bad;
  small_lu_solve<FS_THREADS>(T, M, sh, b, bad);
  if (tid >= 32) return;
#pragma unroll
  for (int s = 0; s < TAPS_MAX_M / 32; ++s)
    if (tid + 32 * s < M) Y[(size_t)i * M + tid + 32 * s] = b[s];
  if (bad && tid == 0) taps_flag(status, TAPS_DEV_SINGULAR);
}

// ---------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------
static bool op_symmetric(int op) { return op != TAPS_OP_G; }
static bool op_mass_like(int op) { return op == TAPS_OP_M || op == TAPS_OP_W; }

// Slot choice of dim d: returns 1 with (slotA, slotB) (slotA = -1 when the dim has a
// single operator) if the dim's distinct operators form a symmetric pencil with a
// mass-like (positive definite) partner.
int taps_fd_eligible(const taps_problem* P, int d, int* slotA, int* slotB) {
  int n = P->tt.nops[d];
  if (n < 1 || n > 2) return 0;
  for (int s = 0; s < n; ++s)
    if (P->ops[d][s] >= TAPS_NUM_OPS) return 0;   // weighted operators: block elimination
  for (int s = 0; s < n; ++s)
    if (!op_symmetric(P->ops[d][s])) return 0;
  if (n == 1) {
    *slotA = -1;
    *slotB = 0;
    return 1;
  }
  int b = op_mass_like(P->ops[d][0]) ? 0 : (op_mass_like(P->ops[d][1]) ? 1 : -1);
  if (b < 0) return 0;
  *slotB = b;
  *slotA = 1 - b;
  return 1;
}

static void fd_pending_free(FdPending& T) {
  cudaFree(T.A);
  memset(&T, 0, sizeof(T));
}

// Cluster size of the tridiagonalisation: 16 CTAs when the device can run a 16-CTA
// cluster of the kernel (non-portable size), else the portable 8.  Both variants do the
// same arithmetic per row and per reduction, so the result does not depend on it.
template <int NC>
static bool td_cluster_ok(const void* fn, size_t smem, int threads) {
  if (NC > 8 && cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  int maxsm = 0, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (taps_allow_dyn_smem(fn, maxsm) != TAPS_OK) {
    cudaGetLastError();
    return false;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(NC);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = NC;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return clusters > 0;
}

template <int NC, typename... Args>
static cudaError_t td_launch(void (*fn)(Args...), int threads, size_t smem, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(NC);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = NC;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, fn, args...);
}

// Whether every SM can hold a CTA of the whole-chip tridiagonalisation.
static bool td_grid_ok(size_t smem, int maxsm) {
  int per_sm = 0;
  if (taps_allow_dyn_smem((const void*)fd_tridiag_grid_kernel, maxsm) != TAPS_OK ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fd_tridiag_grid_kernel, TDG_THREADS, smem) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return per_sm > 0;
}

// The tridiagonalisation of S (n x n in A): S in a cluster's distributed shared memory while its
// rows fit (16 CTAs: n <= 656), then in the shared memory of all num_sms SMs while they fit (152:
// n <= ~1820), else in global memory.  The dim's size alone decides: the decomposition is kept for
// every later solve of the dim, which must not round differently for having come first from a
// batch, and decompositions run side by side from a batch or from a caller's threads as well as
// alone.  Decomposition and first solve of 18 instances in a batch / from 18 threads / of one
// instance, ms, on clusters and on the whole chip: 449 nodes: 49, 93, 9.5 and 114, 122, 9.2; 640:
// 109, 152, 18.8 and 175, 234, 15.0; 800 (a cluster's S in global memory): 225, 376, 41.8 and 251,
// 326, 19.9; 1300: 778, 1073, 123 and 799, 844, 52; 1800: 1916, 2531, 272 and 1774, 1787, 104.
// xch: 4 n doubles and two words of workspace.
static int td_run(double* A, double* V, double* tmp, double* bt, double* dd, double* ee, int n, int maxsm,
                  int num_sms, double* xch, int* status, cudaStream_t s) {
  const size_t dsm16 = sizeof(double) * ((size_t)((n + 15) / 16) * n + 3 * (size_t)n);
  const size_t dsm8 = sizeof(double) * ((size_t)((n + 7) / 8) * n + 3 * (size_t)n);
  const size_t gsm = sizeof(double) * 3 * (size_t)n;
  const size_t grd = sizeof(double) * ((size_t)((n + num_sms - 1) / num_sms) * n + 3 * (size_t)n);
  cudaError_t ce;
  const bool chip = grd + 1024 <= (size_t)maxsm && n <= TDG_THREADS * TDG_PER;
  if (dsm16 + 1024 <= (size_t)maxsm && td_cluster_ok<16>((const void*)fd_tridiag_dsmem_kernel<16>, dsm16, TDS_THREADS)) {
    ce = td_launch<16>(fd_tridiag_dsmem_kernel<16>, TDS_THREADS, dsm16, s, (const double*)A, V, bt, dd, ee, n);
  } else if (dsm8 + 1024 <= (size_t)maxsm && td_cluster_ok<8>((const void*)fd_tridiag_dsmem_kernel<8>, dsm8, TDS_THREADS)) {
    ce = td_launch<8>(fd_tridiag_dsmem_kernel<8>, TDS_THREADS, dsm8, s, (const double*)A, V, bt, dd, ee, n);
  } else if (chip && td_grid_ok(grd, maxsm)) {
    unsigned* bar = reinterpret_cast<unsigned*>(xch + 4 * (size_t)n);
    TAPS_CUDA(cudaMemsetAsync(bar, 0, 2 * sizeof(unsigned), s));
    const double* Ac = A;
    void* args[] = {&Ac, &V, &bt, &dd, &ee, &n, &xch, &bar, &status};
    ce = cudaLaunchCooperativeKernel((const void*)fd_tridiag_grid_kernel, dim3(num_sms), dim3(TDG_THREADS), args, grd, s);
  } else if (td_cluster_ok<16>((const void*)fd_tridiag_kernel<16>, gsm, TD_THREADS)) {
    ce = td_launch<16>(fd_tridiag_kernel<16>, TD_THREADS, gsm, s, A, V, tmp, bt, dd, ee, n);
  } else {
    if (!td_cluster_ok<8>((const void*)fd_tridiag_kernel<8>, gsm, TD_THREADS)) return TAPS_ERR_CUDA;
    ce = td_launch<8>(fd_tridiag_kernel<8>, TD_THREADS, gsm, s, A, V, tmp, bt, dd, ee, n);
  }
  if (ce != cudaSuccess) {
    taps_note_cuda_error(ce, "tridiagonalisation launch", __FILE__, __LINE__);
    return TAPS_ERR_CUDA;
  }
  return TAPS_OK;
}

// The kernels of the half-bandwidths hb = 2 s + 1, s <= TAPS_MAX_S.
template <template <int> class K, typename... Args>
static int fd_by_band(int hb, Args... args) {
  switch (hb) {
    case 1: K<1>::launch(args...); break;
    case 3: K<3>::launch(args...); break;
    case 5: K<5>::launch(args...); break;
    case 7: K<7>::launch(args...); break;
    case 9: K<9>::launch(args...); break;
    default: return TAPS_ERR_INVALID_ARG;
  }
  TAPS_CUDA(cudaGetLastError());
  return TAPS_OK;
}
template <int HB>
struct LsolveLaunch {
  static void launch(const double* L, const double* linv, const double* In, int n, int trans_in, double* Out,
                     cudaStream_t s) {
    fd_lsolve_kernel<HB><<<(n + 31) / 32, 32, 0, s>>>(L, linv, In, n, trans_in, Out);
  }
};
template <int HB>
struct PhiLaunch {
  static void launch(const double* L, const double* linv, const double* Z, const double* lam, int n, double* Phi,
                     double* PhiT, double* mu, int* status, cudaStream_t s) {
    fd_phi_kernel<HB><<<(n + 31) / 32, 32, 0, s>>>(L, linv, Z, lam, n, Phi, PhiT, mu, status);
  }
};
static int fd_lsolve(const double* L, const double* linv, const double* In, int n, int hb, int trans_in, double* Out,
                     cudaStream_t s) {
  return fd_by_band<LsolveLaunch>(hb, L, linv, In, n, trans_in, Out, s);
}
static int fd_phi(const double* L, const double* linv, const double* Z, const double* lam, int n, int hb, double* Phi,
                  double* PhiT, double* mu, int* status, cudaStream_t s) {
  return fd_by_band<PhiLaunch>(hb, L, linv, Z, lam, n, Phi, PhiT, mu, status, s);
}
static int fd_cholesky(const double* band, double* B, int n, int hb, double* linv, int* status, int maxsm,
                       cudaStream_t s) {
  const size_t smem = sizeof(double) * (size_t)n * (hb + 1);
  if (smem + 1024 <= (size_t)maxsm) {
    TAPS_TRY(taps_allow_dyn_smem((const void*)fd_cholesky_kernel, maxsm));
    fd_cholesky_kernel<<<1, 32, smem, s>>>(band, B, n, hb, linv, status);
  } else {
    fd_cholesky_global_kernel<<<1, FD_THREADS, 0, s>>>(B, n, hb, linv, status);
  }
  TAPS_CUDA(cudaGetLastError());
  return TAPS_OK;
}

template <int C>
static int iv_launch(const double* dd, const double* ee, const double* lam, int n, double* Z, int maxsm, cudaStream_t s) {
  TAPS_TRY(taps_allow_dyn_smem((const void*)fd_invit_smem_kernel<C>, maxsm));
  fd_invit_smem_kernel<C><<<(n + C - 1) / C, 32, iv_smem(n, C), s>>>(dd, ee, lam, n, Z);
  return TAPS_OK;
}

// Enqueues the decomposition of the pencil (opA, opB) of dm on P's stream without
// waiting for it: the entry is registered at once (pending, with an event recorded
// after its last kernel) and the temporaries are returned in *T for fd_finish.  An
// entry that already exists, pending on another stream, makes P's stream wait for it.
static int fd_enqueue(taps_problem* P, taps_dim* dm, int opA, int opB, FdEntry** out, FdPending* T) {
  memset(T, 0, sizeof(*T));
  for (int k = 0; k < dm->nfd; ++k)
    if (dm->fd[k].opA == opA && dm->fd[k].opB == opB) {
      *out = &dm->fd[k];
      if (dm->fd[k].pending && dm->fd[k].done) TAPS_CUDA(cudaStreamWaitEvent(P->stream, dm->fd[k].done, 0));
      return dm->fd[k].status;
    }
  if (dm->nfd >= 4) return TAPS_ERR_INVALID_ARG;
  FdEntry& E = dm->fd[dm->nfd];
  memset(&E, 0, sizeof(E));
  E.opA = opA;
  E.opB = opB;
  int n = dm->nf;
  size_t nn = (size_t)n * n;
  cudaStream_t s = P->stream;
  const int hasA = opA >= 0 ? 1 : 0;
  int st = TAPS_OK;
  T->E = &E;
  T->P = P;
  do {
    // the back-transform keeps one column per warp in shared memory (n <= 6144); the
    // tridiagonalisation stages three vectors (3n doubles)
    if (sizeof(double) * (size_t)n > 48 * 1024) { st = TAPS_ERR_INVALID_ARG; break; }
    int maxsm_optin = 0;
    {
      int dev = 0;
      cudaGetDevice(&dev);
      cudaDeviceGetAttribute(&maxsm_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    }
    if ((st = taps_alloc((void**)&E.Phi, sizeof(double) * nn)) != TAPS_OK) break;
    if ((st = taps_alloc((void**)&E.PhiT, sizeof(double) * nn)) != TAPS_OK) break;
    if ((st = taps_alloc((void**)&E.mu, sizeof(double) * n)) != TAPS_OK) break;
    // eigenvectors to a CTA of the inverse iteration: as many as fit its shared memory, 0 for the
    // kernel on global arrays
    int cols = 8;
    while (cols > 0 && iv_smem(n, cols) + 1024 > (size_t)maxsm_optin) cols >>= 1;
    {
      const size_t nW = hasA ? (cols == 0 ? 5 : 2) * nn : 0;
      if ((st = taps_alloc((void**)&T->A, sizeof(double) * (3 * nn + nW + 6 * (size_t)n))) != TAPS_OK) break;
      T->B = T->A + nn;
      T->V = T->B + nn;
      T->tmp = T->V + nn;
      T->bt = T->tmp + 2 * n;
      T->dd = T->bt + n;
      T->ee = T->dd + n;
      T->lam = T->ee + n;
      T->W = T->lam + n;
    }
    double *A = T->A, *B = T->B, *V = T->V, *W = T->W, *lam = T->lam;
    const size_t bsz = (size_t)n * dm->nb;
    const double* bandA = hasA ? dm->d_band + (size_t)opA * bsz : nullptr;
    const double* bandB = dm->d_band + (size_t)opB * bsz;
    int tk = prof_begin(P, TAPS_PROF_OTHER);
    fd_dense_kernel<<<(unsigned)((nn + 255) / 256), 256, 0, s>>>(bandA, bandB, n, dm->hb, A, B);
    if (cudaMemsetAsync(V, 0, sizeof(double) * nn, s) != cudaSuccess) { st = TAPS_ERR_CUDA; break; }
    // banded Cholesky and S, then the tridiagonalisation
    double* linv = T->tmp + n;   // the tridiagonalisation uses the first n
    if ((st = fd_cholesky(bandB, B, n, dm->hb, linv, P->d_status, maxsm_optin, s)) != TAPS_OK) break;
    if (hasA) {
      // S = L^{-1} A L^{-T}: X = L^{-1} A into V, S^T = L^{-1} X^T into W, symmetrised into A
      if ((st = fd_lsolve(B, linv, A, n, dm->hb, 0, V, s)) != TAPS_OK) break;
      if ((st = fd_lsolve(B, linv, V, n, dm->hb, 1, W, s)) != TAPS_OK) break;
      fd_symmetrize_kernel<<<(unsigned)((nn + 255) / 256), 256, 0, s>>>(W, n, A);
      if (cudaMemsetAsync(V, 0, sizeof(double) * nn, s) != cudaSuccess) { st = TAPS_ERR_CUDA; break; }
      if ((st = td_run(A, V, T->tmp, T->bt, T->dd, T->ee, n, maxsm_optin, P->num_sms, W, P->d_status, s)) != TAPS_OK) break;
      // eigenvalues (warp each), eigenvectors (thread each), back-transform (warp each),
      // all into A, which the tridiagonalisation no longer needs
      // two warps per CTA: the warps' FP64 chains spread over the SMs' sub-partitions
      if ((st = taps_allow_dyn_smem((const void*)fd_bisect_kernel, maxsm_optin)) != TAPS_OK) break;
      fd_bisect_kernel<<<(unsigned)((32LL * n + 63) / 64), 64, sizeof(double) * 2 * n, s>>>(T->dd, T->ee, n, lam);
      // eigenvectors in shared memory, as many to a CTA as fit, else one thread per eigenvector
      // on global arrays, in 32-thread CTAs: the chains spread over the SMs
      if (cols == 8) st = iv_launch<8>(T->dd, T->ee, lam, n, A, maxsm_optin, s);
      else if (cols == 4) st = iv_launch<4>(T->dd, T->ee, lam, n, A, maxsm_optin, s);
      else if (cols == 2) st = iv_launch<2>(T->dd, T->ee, lam, n, A, maxsm_optin, s);
      else if (cols == 1) st = iv_launch<1>(T->dd, T->ee, lam, n, A, maxsm_optin, s);
      if (st != TAPS_OK) break;
      if (cols == 0) {
        fd_invit_kernel<<<(n + 31) / 32, 32, 0, s>>>(T->dd, T->ee, lam, n, A, W);
      }
      // symmetric orthogonalisation: E in W, the corrected vectors back into A
      const unsigned gnn = (unsigned)((nn + 255) / 256);
      fd_gram_minus_identity_kernel<<<gnn, 256, 0, s>>>(A, n, W);
      fd_orth_update_kernel<<<gnn, 256, 0, s>>>(A, W, n, W + nn);
      if (cudaMemcpyAsync(A, W + nn, sizeof(double) * nn, cudaMemcpyDeviceToDevice, s) != cudaSuccess) {
        st = TAPS_ERR_CUDA;
        break;
      }
      // few warps per CTA: one to an SM sub-partition while the columns fit the chip that way
      const int most = std::max(1, std::min(8, (int)(48 * 1024 / (sizeof(double) * (size_t)n))));
      const int wpc = std::min(most, std::max(1, (n + P->num_sms - 1) / P->num_sms));
      fd_backtransform_kernel<<<(n + wpc - 1) / wpc, 32 * wpc, sizeof(double) * (size_t)n * wpc, s>>>(
          V, T->bt, n, A);
    }
    if ((st = fd_phi(B, linv, hasA ? A : nullptr, hasA ? lam : nullptr, n, dm->hb, E.Phi, E.PhiT, E.mu, P->d_status,
                     s)) != TAPS_OK)
      break;
    prof_end(P, TAPS_PROF_OTHER, tk, (10.0 / 3.0) * (double)nn * n, 8.0 * 4.0 * nn);
    cudaError_t ce = cudaGetLastError();
    if (ce != cudaSuccess) {
      taps_note_cuda_error(ce, "pencil decomposition", __FILE__, __LINE__);
      st = TAPS_ERR_CUDA;
      break;
    }
    if (cudaEventCreateWithFlags(&E.done, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventRecord(E.done, s) != cudaSuccess) {
      st = TAPS_ERR_CUDA;
      break;
    }
  } while (0);
  E.status = st;
  E.pending = (st == TAPS_OK) ? 1 : 0;
  dm->nfd++;
  *out = &E;
  if (st != TAPS_OK) fd_pending_free(*T);
  return st;
}

// Waits for a decomposition enqueued by fd_enqueue, reads its problem's device status
// into the entry and frees the temporaries.
static int fd_finish(FdPending& T) {
  if (!T.E) return TAPS_OK;
  int st = taps_check_status(T.P->d_status, T.P->stream);
  if (T.E->status == TAPS_OK) T.E->status = st;
  T.E->pending = 0;
  if (T.E->done) {
    cudaEventDestroy(T.E->done);
    T.E->done = nullptr;
  }
  fd_pending_free(T);
  return st;
}

static int fd_prepare(taps_problem* P, int d, taps_dim* dm, int opA, int opB, FdEntry** out) {
  (void)d;
  FdPending T;
  int st = fd_enqueue(P, dm, opA, opB, out, &T);
  if (st != TAPS_OK) return st;
  return fd_finish(T);
}

// Reduced solve of dim d by fast diagonalisation, coefficients in P->d_C / P->d_c.
int taps_fd_solve(taps_problem* P, taps_factors* U, int d, int precision) {
  int slotA, slotB;
  if (!taps_fd_eligible(P, d, &slotA, &slotB)) return TAPS_ERR_INVALID_ARG;
  taps_dim* dm = P->dims[d];
  FdEntry* E = nullptr;
  int opA = slotA >= 0 ? P->ops[d][slotA] : -1;
  TAPS_TRY(fd_prepare(P, d, dm, opA, P->ops[d][slotB], &E));
  if (!P->d_pq[d]) return TAPS_ERR_INVALID_ARG;   // taps_fd_prepare_all comes first
  const int n = dm->nf, M = U->M;
  const size_t MM = (size_t)M * M;
  cudaStream_t s = P->stream;
  const int nM = n * M;
  double* G = P->d_Y;
  double* Y = P->d_Y + (size_t)n * M;
  int tk = prof_begin(P, TAPS_PROF_FASTDIAG);
  const double* CA = slotA >= 0 ? P->d_C + (size_t)slotA * MM : nullptr;
  const double* CB = P->d_C + (size_t)slotB * MM;
  int launches = 2;
  if (M <= 32 && precision != TAPS_MIXED) {
    TAPS_CUDA(taps_launch_pdl(fd_small_solve_quad_kernel, dim3(n), dim3(128), 0, s, CA, CB,
                              slotA >= 0 ? (const double*)E->mu : nullptr, (const double*)P->d_pq[d],
                              (const double*)P->d_c, P->Rf, n, M, Y, P->d_status));
  } else {
    TAPS_TRY(taps_rhs(P->d_pq[d], P->d_c, P->Rf, n, M, G, P->num_sms, s));
    if (M <= 32)
      fd_small_solve_warp_kernel<<<n, 32, 0, s>>>(CA, CB, slotA >= 0 ? E->mu : nullptr, G, n, M, Y,
                                                  P->d_status, 1);
    else {
      // M (M + 1) doubles exceed the default 48 KB from M = 78 on: allow up to M = 128
      static bool smem_ok = false;
      if (!smem_ok) {
        int dev = 0, maxsm = 0;
        TAPS_CUDA(cudaGetDevice(&dev));
        TAPS_CUDA(cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
        TAPS_TRY(taps_allow_dyn_smem((const void*)fd_small_solve_kernel, maxsm));
        smem_ok = true;
      }
      fd_small_solve_kernel<<<n, FS_THREADS, sizeof(double) * (size_t)M * (M + 1), s>>>(
          CA, CB, slotA >= 0 ? E->mu : nullptr, G, M, Y, P->d_status);
    }
    ++launches;
  }
  P->prof->launches[TAPS_PROF_FASTDIAG] += launches - 2;
  prof_end(P, TAPS_PROF_FASTDIAG, tk, 2.0 * P->Rf * nM + n * ((2.0 / 3.0) * M * MM + 2.0 * MM),
           8.0 * ((double)P->Rf * n + 2.0 * MM + (double)nM));
  // back to the nodal basis; the previous factor goes to d_Uold for the change norm
  tk = prof_begin(P, TAPS_PROF_FD_TRANSFORM);
  TAPS_TRY(fd_transform(E->Phi, Y, n, M, U->d_U[d], 1, P->d_Uold, s));
  prof_end(P, TAPS_PROF_FD_TRANSFORM, tk, 2.0 * (double)n * n * M, 8.0 * ((double)n * n + 3.0 * nM));
  TAPS_CUDA(cudaGetLastError());
  return TAPS_OK;
}

// The cached (or newly made) decomposition of the pencil (opA, opB) of dim d.
int taps_fd_lookup(taps_problem* P, int d, int opA, int opB, const FdEntry** out) {
  FdEntry* E = nullptr;
  TAPS_TRY(fd_prepare(P, d, P->dims[d], opA, opB, &E));
  *out = E;
  return TAPS_OK;
}

// Out = Phi Y in the factor layout (Y n x M row-major), the previous factor into Save.
int taps_fd_to_nodal(taps_problem* P, const FdEntry* E, const double* Y, int n, int M, double* Out, double* Save) {
  int tk = prof_begin(P, TAPS_PROF_FD_TRANSFORM);
  TAPS_TRY(fd_transform(E->Phi, Y, n, M, Out, 1, Save, P->stream));
  prof_end(P, TAPS_PROF_FD_TRANSFORM, tk, 2.0 * (double)n * n * M, 8.0 * ((double)n * n + 3.0 * (double)n * M));
  TAPS_CUDA(cudaGetLastError());
  return TAPS_OK;
}

// Pencil decompositions of every eligible dim, done before any capture (they
// allocate and synchronise).  The enqueue half launches them on P's stream and keeps
// their temporaries in *pend; the finish half waits, checks and frees.  Batches
// enqueue many problems (each on its own stream) before finishing any, so the
// decompositions of different instances run concurrently.
int taps_fd_prepare_enqueue(taps_problem* P, int solver, int M, std::vector<FdPending>* pend) {
  if (solver != TAPS_SOLVER_FASTDIAG && solver != TAPS_SOLVER_MODEDIAG) return TAPS_OK;
  for (int d = 0; d < P->D; ++d) {
    int sa, sb;
    const int route = taps_dim_route(P, d, solver, M);
    if (route == TAPS_ROUTE_FDW) {
      int s0, s1, nb;
      taps_fdw_eligible(P, d, M, &sa, &sb, &s0, &s1, &nb);
    } else if (route != TAPS_ROUTE_FD || !taps_fd_eligible(P, d, &sa, &sb)) {
      continue;
    }
    FdEntry* E = nullptr;
    FdPending T;
    TAPS_TRY(fd_enqueue(P, P->dims[d], sa >= 0 ? P->ops[d][sa] : -1, P->ops[d][sb], &E, &T));
    if (T.E) pend->push_back(T);
    if (!P->d_pq[d]) {   // the problem's source vectors in the pencil's eigenbasis
      const int n = P->dims[d]->nf;
      const long long tot = (long long)n * P->Rf;
      TAPS_TRY(taps_alloc((void**)&P->d_pq[d], sizeof(double) * (size_t)std::max(tot, 1LL)));
      if (tot > 0)
        fd_pq_kernel<<<(unsigned)((tot + 127) / 128), 128, 0, P->stream>>>(E->Phi, P->d_q[d], n, P->Rf,
                                                                           P->d_pq[d]);
      TAPS_CUDA(cudaGetLastError());
    }
  }
  return TAPS_OK;
}

int taps_fd_prepare_finish(std::vector<FdPending>* pend) {
  int st = TAPS_OK;
  for (auto& T : *pend) {
    int s2 = fd_finish(T);
    if (st == TAPS_OK) st = s2;
  }
  pend->clear();
  return st;
}

int taps_fd_prepare_all(taps_problem* P, int solver, int M) {
  std::vector<FdPending> pend;
  int st = taps_fd_prepare_enqueue(P, solver, M, &pend);
  int s2 = taps_fd_prepare_finish(&pend);
  return st != TAPS_OK ? st : s2;
}

void taps_fd_release(taps_dim* dm) {
  for (int k = 0; k < dm->nfd; ++k) {
    cudaFree(dm->fd[k].Phi);
    cudaFree(dm->fd[k].PhiT);
    cudaFree(dm->fd[k].mu);
    if (dm->fd[k].done) cudaEventDestroy(dm->fd[k].done);
  }
  dm->nfd = 0;
}

// ---------------------------------------------------------------------------------
// The small solves' reciprocal on a device array (for checking it against IEEE
// division).
// ---------------------------------------------------------------------------------
__global__ void rcp_kernel(const double* __restrict__ x, double* __restrict__ y, long long n) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = taps_rcp(x[i]);
}

extern "C" int taps_util_rcp(const double* x_dev, double* y_dev, long long n, void* stream) {
  if (n < 0 || (n > 0 && (!x_dev || !y_dev))) return TAPS_ERR_INVALID_ARG;
  if (n == 0) return TAPS_OK;
  rcp_kernel<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream>>>(x_dev, y_dev, n);
  TAPS_CUDA(cudaGetLastError());
  return TAPS_OK;
}

// ---------------------------------------------------------------------------------
// The library's bounded grid barrier with a short poll limit, for its failure test:
// `ctas` CTAs meet at a barrier that expects ctas + missing arrivals, twice.  With
// missing > 0 every wait runs out after `limit` polls, records TAPS_DEV_TIMEOUT and the
// kernel returns; the host reads the status.  Nothing waits without a bound.
// ---------------------------------------------------------------------------------
__global__ void barrier_test_kernel(unsigned* bar, int* status, unsigned expected, long long limit) {
  grid_barrier(bar, status, expected, limit);
  grid_barrier(bar, status, expected, limit);
}

extern "C" int taps_util_barrier_test(int ctas, int missing, long long poll_limit, void* stream) {
  if (ctas < 1 || ctas > 64 || missing < 0 || missing > 64 || poll_limit < 1 || poll_limit > (1ll << 26))
    return TAPS_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  unsigned* bar = nullptr;
  int* status = nullptr;
  TAPS_TRY(taps_alloc((void**)&bar, 2 * sizeof(unsigned)));
  if (taps_alloc((void**)&status, sizeof(int)) != TAPS_OK) {
    cudaFree(bar);
    return TAPS_ERR_OOM;
  }
  int st = TAPS_OK;
  if (cudaMemsetAsync(bar, 0, 2 * sizeof(unsigned), s) != cudaSuccess ||
      cudaMemsetAsync(status, 0, sizeof(int), s) != cudaSuccess) {
    st = TAPS_ERR_CUDA;
  } else {
    barrier_test_kernel<<<ctas, 32, 0, s>>>(bar, status, (unsigned)(ctas + missing), poll_limit);
    if (cudaGetLastError() != cudaSuccess) st = TAPS_ERR_CUDA;
    else st = taps_check_status(status, s);
  }
  cudaStreamSynchronize(s);
  cudaFree(bar);
  cudaFree(status);
  return st;
}
