// Node-side diagonalisation of a dimension with convection faces (Sec. 2.6 route,
// extended to the point-mass terms of Eqs. 21/25).
//
// A space dim with convection faces has, besides its stiffness A (K) and mass B (M or
// W), one or two point-mass operators beta_b e_b e_b^T at its end nodes b.  With the
// pencil basis Phi (Phi^T B Phi = I, Phi^T A Phi = diag(mu)) and U = Phi Y, row i of the
// reduced system reads
//     T_i y_i + sum_b beta_b phi_b[i] C_b z_b = g_i,   z_b = sum_j phi_b[j] y_j,
// with T_i = mu_i C_A + C_B, g_i = (Phi^T F)[i], phi_b = Phi^T e_b (row b of Phi) and
// C_b the coefficient matrix of face b's operator.  The face terms couple the nodes
// only through the nb M-vectors z_b, so (Sherman-Morrison-Woodbury)
//     y_i = w_i - T_i^-1 sum_b beta_b phi_b[i] C_b z_b,   w_i = T_i^-1 g_i,
// and the z_b solve the (nb M) x (nb M) capacitance system
//     z_b' + sum_b beta_b (sum_i phi_b'[i] phi_b[i] T_i^-1) C_b z_b = sum_i phi_b'[i] w_i.
//
//   (taps_rhs)         g_i = sum_r (Phi^T q_r)[i] c_r for every node.
//   fdw_node_kernel    four warps per node: LU of T_i without pivoting, w_i and T_i^-1
//                      (1 + M right-hand sides, lane = row).
//   fdw_reduce_kernel  the sums over the nodes: Z_b'b = sum_i phi_b' phi_b T_i^-1 and
//                      the capacitance right-hand side.
//   fdw_cap_kernel     one CTA: the capacitance blocks Z_b'b C_b and their system by LU with
//                      partial pivoting, then u_b = C_b z_b.
//   fdw_final_kernel   y_i; then the node-side transform U = Phi Y (fd_rowgemm_kernel).
#include <string.h>

#include <algorithm>

#include "small_lu.cuh"
#include "taps_internal.cuh"

// One CTA of four warps per node (M <= 32): T_i = mu_i C_A + C_B factored as L U without
// pivoting (the symmetric part of T_i is positive definite), then w_i = T_i^-1 g_i and T_i^-1.
// A warp-wide FP64 instruction holds its SM sub-partition ~64 cycles whatever lanes it uses, so
// the issue of the M^3-sized work is the bound and it is spread over the four sub-partitions:
// role w holds the columns c = w, w + 4, ... (lane = row), of T_i first and of the identity
// after, and the role with the fewest columns takes g_i.  The multipliers and U go to shared
// memory column by column.  Columns of L^-1 start at their own row; a backward step's M / 4
// products with the pivot's reciprocal are one multiplication across lanes.  CTAs num_sms apart,
// which land on one SM, put the same role on different sub-partitions.  255 nodes of 20 modes:
// 125 us with one warp per node, 36 us now.
__global__ void __launch_bounds__(128) fdw_node_kernel(const double* __restrict__ CA, const double* __restrict__ CB,
                                                       const double* __restrict__ mu, const double* __restrict__ G,
                                                       int n, int M, int num_sms, double* __restrict__ X,
                                                       double* __restrict__ w, int* status) {
  __shared__ double LU[32][33];   // [column][row]: multipliers below the diagonal, U on and above it
  __shared__ double invd[32];
  const int i = blockIdx.x, lane = threadIdx.x & 31;
  const int role = ((threadIdx.x >> 5) + 2 * (i / num_sms)) & 3;
  const bool act = lane < M;
  const double mi = mu[i];
  double v[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int c = 4 * k + role;
    v[k] = (act && c < M) ? fma(mi, CA[lane * M + c], CB[lane * M + c]) : 0.0;
  }
  double g = (role == (M & 3) && act) ? G[(size_t)i * M + lane] : 0.0;
  bool bad = false;
  // the multipliers of a step and the pivot's reciprocal (0 for a zero or non-finite pivot)
  auto publish = [&](int q, double col, double piv) {
    const bool ok = taps_finite_nonzero(piv);
    bad |= !ok;
    const double ip = ok ? taps_rcp(piv) : 0.0;
    LU[q][lane] = (lane > q && act) ? col * ip : 0.0;
    if (lane == 0) invd[q] = ip;
  };
  if (role == 0) publish(0, v[0], __shfl_sync(0xffffffffu, v[0], 0));
  __syncthreads();
#pragma unroll
  for (int p = 0; p < 32; ++p) {
    if (p < M) {
      const double l = LU[p][lane];
      const int q = p + 1;   // next pivot column, owned by role q & 3 in slot q >> 2
      const bool owner = q < M && role == (q & 3);
      if (owner) {
        v[(q >> 2) & 7] -= l * __shfl_sync(0xffffffffu, v[(q >> 2) & 7], p);
        publish(q, v[(q >> 2) & 7], __shfl_sync(0xffffffffu, v[(q >> 2) & 7], q & 31));
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) {   // this role's columns c > p
        const int c = 4 * k + role;
        if (4 * k + 3 <= p || c <= p || c >= M || (owner && c == q)) continue;
        v[k] -= l * __shfl_sync(0xffffffffu, v[k], p);
      }
      __syncthreads();
    }
  }
  if (bad && lane == 0) taps_flag(status, TAPS_DEV_SINGULAR);
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int c = 4 * k + role;
    if (c < M && lane <= c) LU[c][lane] = v[k];
  }
  __syncthreads();
  // columns of the identity (and g): forward from the column's own row, then backward
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = (act && lane == 4 * k + role) ? 1.0 : 0.0;
  const bool has_g = role == (M & 3);
  for (int p = 0; p < M; ++p) {
    const double l = LU[p][lane];
    if (has_g) {
      const double t = __shfl_sync(0xffffffffu, g, p);
      if (lane > p) g -= l * t;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int c = 4 * k + role;
      if (c > p || c >= M) continue;
      const double t = __shfl_sync(0xffffffffu, v[k], p);
      if (lane > p) v[k] -= l * t;
    }
  }
  for (int p = M - 1; p >= 0; --p) {
    const double u = LU[p][lane];
    double xp = has_g ? __shfl_sync(0xffffffffu, g, p) : 0.0;   // row p of slot k in lane k, of g in lane 8
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (4 * k + role >= M) continue;
      const double t = __shfl_sync(0xffffffffu, v[k], p);
      if (lane == k) xp = t;
    }
    xp *= invd[p];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (4 * k + role >= M) continue;
      const double t = __shfl_sync(0xffffffffu, xp, k);
      if (lane == p) v[k] = t;
      if (lane < p) v[k] -= u * t;
    }
    if (has_g) {
      const double t = __shfl_sync(0xffffffffu, xp, 8);
      if (lane == p) g = t;
      if (lane < p) g -= u * t;
    }
  }
  if (has_g && act) w[(size_t)i * M + lane] = g;
  // T_i^-1 row by row through shared memory (whole-sector stores)
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 8; ++k)
    if (4 * k + role < M) LU[4 * k + role][lane] = v[k];
  __syncthreads();
  for (int idx = threadIdx.x; idx < M * M; idx += 128) X[(size_t)i * M * M + idx] = LU[idx % M][idx / M];
}

// Z[b'][b][r][c] = sum_i phi_b'[i] phi_b[i] T_i^-1[r][c];  rr[b'][r] = sum_i phi_b'[i] w_i[r].
// phi_b[i] = Phi[corner_b][i] (row corner_b of Phi: Phi^T e_b).  X holds T_i^-1.
// blockIdx.y = the pair (b', b), b' <= b (the weights of (b, b') are the same), then the rows
// of rr; one warp adds 32 entries over the nodes in order, the products of phi formed once per
// CTA in shared memory.  The chain of n FMAs is the bound: 255 nodes of 20 modes, two faces,
// 34 us with the products in every thread and all four pairs, 23 us now.
#define FDW_RED_NODES 512
__global__ void __launch_bounds__(32) fdw_reduce_kernel(const double* __restrict__ X, const double* __restrict__ w,
                                                        const double* __restrict__ Phi, int c0, int c1, int n, int M,
                                                        int nbnd, double* __restrict__ Z, double* __restrict__ rr) {
  __shared__ double ph[FDW_RED_NODES];
  const int e = blockIdx.x * 32 + threadIdx.x, MM = M * M;
  const int npair = nbnd == 2 ? 3 : 1;
  const bool pair = (int)blockIdx.y < npair;
  const int q = pair ? blockIdx.y : blockIdx.y - npair;
  const int bp = pair ? q >> 1 : q, b = pair ? (q + 1) >> 1 : q;   // (0,0), (0,1), (1,1)
  const int count = pair ? MM : M;
  if ((int)blockIdx.x * 32 >= count) return;
  const double* pb = Phi + (size_t)(b == 0 ? c0 : c1) * n;
  const double* pbp = Phi + (size_t)(bp == 0 ? c0 : c1) * n;
  const double* src = pair ? X : w;
  const int ec = min(e, count - 1);
  double v = 0.0;
  for (int i0 = 0; i0 < n; i0 += FDW_RED_NODES) {
    const int len = min(FDW_RED_NODES, n - i0);
    __syncwarp();
    for (int i = threadIdx.x; i < len; i += 32) ph[i] = pair ? pbp[i0 + i] * pb[i0 + i] : pbp[i0 + i];
    __syncwarp();
    const double* xs = src + (size_t)i0 * count + ec;
    v = taps_fma_chain<16>(
        len, [&](int i) { return ph[i]; }, [&](int i) { return xs[(size_t)i * count]; }, v);
  }
  if (e >= count) return;
  if (!pair) {
    rr[bp * M + e] = v;
    return;
  }
  Z[(size_t)(bp * nbnd + b) * MM + e] = v;
  if (b != bp) Z[(size_t)(b * nbnd + bp) * MM + e] = v;
}

// (I + [beta_b Z[b'][b] C_b]) z = rr, N2 = nbnd M <= 64 unknowns, partial pivoting; beta_b
// is the corner entry of face b's point-mass band.  Writes u_b = C_b z_b and beta for the
// final kernel.
// One CTA (small_lu.cuh: the pivot search of a single thread, a row per thread and a single
// thread's back substitution took 150 us for 40 unknowns).
#define FDW_MAXN 64
#define FDW_CAP_THREADS 256
__global__ void __launch_bounds__(FDW_CAP_THREADS) fdw_cap_kernel(const double* __restrict__ Z, const double* __restrict__ rr,
                                                     const double* __restrict__ band0,
                                                     const double* __restrict__ band1, int corner0, int corner1,
                                                     int hb, int M, int nbnd, const double* __restrict__ C0,
                                                     const double* __restrict__ C1, double* __restrict__ z,
                                                     double* __restrict__ beta, int* status) {
  __shared__ double A[FDW_MAXN * (FDW_MAXN + 1)];
  __shared__ SmallLu sh;
  __shared__ double bet[2], zs[FDW_MAXN];
  const int tid = threadIdx.x, N2 = nbnd * M, nb = 2 * hb + 1, ld = N2 + 1;
  if (tid < nbnd) {
    const double* bd = tid == 0 ? band0 : band1;
    const int cr = tid == 0 ? corner0 : corner1;
    bet[tid] = bd[(size_t)cr * nb + hb];
  }
  __syncthreads();
  // Z into the matrix's place, the products Z[b'][b] C_b in registers, then the matrix
  for (int idx = tid; idx < N2 * N2; idx += FDW_CAP_THREADS) {
    const int rI = idx / N2, cI = idx % N2;
    const int bp = rI / M, r = rI % M, b = cI / M, cc = cI % M;
    A[rI * ld + cI] = Z[(((size_t)bp * nbnd + b) * M + r) * M + cc];
  }
  __syncthreads();
  constexpr int PER = FDW_MAXN * FDW_MAXN / FDW_CAP_THREADS;
  double v[PER];
#pragma unroll
  for (int e = 0; e < PER; ++e) {
    const int idx = tid + e * FDW_CAP_THREADS;
    if (idx >= N2 * N2) break;
    const int rI = idx / N2, cI = idx % N2, b = cI / M, cc = cI % M;
    const double* Cb = b == 0 ? C0 : C1;
    const double* zr = A + rI * ld + b * M;
    double sum = 0.0;
#pragma unroll 4
    for (int k = 0; k < M; ++k) sum = fma(zr[k], Cb[(size_t)k * M + cc], sum);
    v[e] = (rI == cI ? 1.0 : 0.0) + bet[b] * sum;
  }
  __syncthreads();
#pragma unroll
  for (int e = 0; e < PER; ++e) {
    const int idx = tid + e * FDW_CAP_THREADS;
    if (idx >= N2 * N2) break;
    A[idx / N2 * ld + idx % N2] = v[e];
  }
  for (int rI = tid; rI < N2; rI += FDW_CAP_THREADS) A[rI * ld + N2] = rr[rI];
  if (tid < nbnd) beta[tid] = bet[tid];
  double x[TAPS_MAX_M / 32];
  bool bad;
  small_lu_solve<FDW_CAP_THREADS>(A, N2, sh, x, bad);
  if (tid < 32) {
#pragma unroll
    for (int s = 0; s < FDW_MAXN / 32; ++s)
      if (tid + 32 * s < N2) zs[tid + 32 * s] = x[s];
    if (bad && tid == 0) taps_flag(status, TAPS_DEV_SINGULAR);
  }
  __syncthreads();
  // u_b = C_b z_b, stored in z's place (the final kernel needs only u)
  for (int rI = tid; rI < N2; rI += FDW_CAP_THREADS) {
    const int b = rI / M, r = rI % M;
    const double* Cb = b == 0 ? C0 : C1;
    double u = 0.0;
    for (int k = 0; k < M; ++k) u = fma(Cb[(size_t)r * M + k], zs[b * M + k], u);
    z[rI] = u;
  }
}

// Y[i][r] = w_i[r] - (T_i^-1 v_i)[r],  v_i = sum_b beta_b phi_b[i] u_b   (row-major n x M)
__global__ void fdw_final_kernel(const double* __restrict__ X, const double* __restrict__ w,
                                 const double* __restrict__ u, const double* __restrict__ beta,
                                 const double* __restrict__ Phi, int c0, int c1, int n, int M, int nbnd,
                                 double* __restrict__ Y) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)n * M) return;
  const int r = (int)(idx % M), i = (int)(idx / M);
  const double f0 = beta[0] * Phi[(size_t)c0 * n + i];
  const double f1 = nbnd > 1 ? beta[1] * Phi[(size_t)c1 * n + i] : 0.0;
  const double* x = X + ((size_t)i * M + r) * M;
  double s = 0.0;
  for (int k = 0; k < M; ++k) {
    const double v = nbnd > 1 ? fma(f1, u[M + k], f0 * u[k]) : f0 * u[k];
    s = fma(x[k], v, s);
  }
  Y[idx] = w[idx] - s;
}

// ---------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------
int taps_fdw_eligible(const taps_problem* P, int d, int M, int* slotA, int* slotB, int* slotC0, int* slotC1,
                      int* nbnd) {
  const int nops = P->tt.nops[d];
  if (nops < 3 || nops > 4 || M < 1 || M > 32) return 0;
  int a = -1, b = -1, lo = -1, hi = -1;
  for (int s = 0; s < nops; ++s) {
    const int op = P->ops[d][s];
    if (op == TAPS_OP_BLO) {
      if (lo >= 0) return 0;
      lo = s;
    } else if (op == TAPS_OP_BHI) {
      if (hi >= 0) return 0;
      hi = s;
    } else if (op == TAPS_OP_M || op == TAPS_OP_W) {
      if (b >= 0) return 0;
      b = s;
    } else if (op == TAPS_OP_K) {
      if (a >= 0) return 0;
      a = s;
    } else {
      return 0;
    }
  }
  if (a < 0 || b < 0 || (lo < 0 && hi < 0)) return 0;
  *slotA = a;
  *slotB = b;
  *nbnd = 0;
  *slotC0 = *slotC1 = -1;
  if (lo >= 0) *(((*nbnd)++ == 0) ? slotC0 : slotC1) = lo;
  if (hi >= 0) *(((*nbnd)++ == 0) ? slotC0 : slotC1) = hi;
  return 1;
}

// T_i^-1 [nf_max][M][M], w [nf_max][M], Z [4][M][M], rr, z / u, beta.
size_t taps_fdw_scratch_doubles(int nf_max, int M) {
  return (size_t)nf_max * ((size_t)M * M + M) + 4 * (size_t)M * M + 4 * (size_t)M + 8;
}

// Reduced solve of dim d (coefficients in P->d_C / P->d_c) through the pencil of its
// stiffness and mass operators; the previous factor goes to P->d_Uold.
int taps_fdw_solve(taps_problem* P, taps_factors* U, int d) {
  int sa, sb, s0, s1, nbnd;
  const int M = U->M;
  if (!taps_fdw_eligible(P, d, M, &sa, &sb, &s0, &s1, &nbnd) || !P->d_fdw || !P->d_pq[d])
    return TAPS_ERR_INVALID_ARG;
  const FdEntry* E = nullptr;
  TAPS_TRY(taps_fd_lookup(P, d, P->ops[d][sa], P->ops[d][sb], &E));
  const taps_dim* dm = P->dims[d];
  const int n = dm->nf, hb = dm->hb;
  const size_t MM = (size_t)M * M;
  cudaStream_t s = P->stream;
  double* X = P->d_fdw;                        // T_i^-1
  double* w = X + (size_t)P->nf_max * MM;
  double* Z = w + (size_t)P->nf_max * M;
  double* rr = Z + 4 * MM;
  double* z = rr + 2 * (size_t)M;
  double* beta = z + 2 * (size_t)M;
  double* Y = P->d_Y + (size_t)n * M;
  const int k0 = P->ops[d][s0], k1 = s1 >= 0 ? P->ops[d][s1] : k0;
  const int corner0 = k0 == TAPS_OP_BLO ? 0 : n - 1, corner1 = k1 == TAPS_OP_BLO ? 0 : n - 1;
  const size_t bsz = (size_t)n * dm->nb;
  const double* C0 = P->d_C + (size_t)s0 * MM;
  const double* C1 = s1 >= 0 ? P->d_C + (size_t)s1 * MM : C0;
  int tk = prof_begin(P, TAPS_PROF_FASTDIAG);
  // g_i for every node first: inside the node's one warp, hundreds of source terms' loads were
  // most of its time
  TAPS_TRY(taps_rhs(P->d_pq[d], P->d_c, P->Rf, n, M, P->d_Y, P->num_sms, s));
  fdw_node_kernel<<<n, 128, 0, s>>>(P->d_C + (size_t)sa * MM, P->d_C + (size_t)sb * MM, E->mu, P->d_Y, n, M,
                                    P->num_sms, X, w, P->d_status);
  fdw_reduce_kernel<<<dim3((M * M + 31) / 32, nbnd == 2 ? 5 : 2), 32, 0, s>>>(X, w, E->Phi, corner0, corner1, n, M,
                                                                              nbnd, Z, rr);
  fdw_cap_kernel<<<1, FDW_CAP_THREADS, 0, s>>>(Z, rr, dm->d_band + (size_t)k0 * bsz, dm->d_band + (size_t)k1 * bsz, corner0,
                                  corner1, hb, M, nbnd, C0, C1, z, beta, P->d_status);
  const long long nM = (long long)n * M;
  fdw_final_kernel<<<(unsigned)((nM + 255) / 256), 256, 0, s>>>(X, w, z, beta, E->Phi, corner0, corner1, n, M,
                                                                 nbnd, Y);
  P->prof->launches[TAPS_PROF_FASTDIAG] += 4;
  const double Md = M;
  prof_end(P, TAPS_PROF_FASTDIAG, tk,
           n * ((2.0 / 3.0) * Md * Md * Md + (1.0 + Md) * 2.0 * Md * Md + 2.0 * P->Rf * Md) +
               2.0 * n * (nbnd * nbnd * (double)MM + nbnd * Md) + 2.0 * nbnd * nbnd * (double)MM * Md +
               (2.0 / 3.0) * pow(nbnd * Md, 3) + 2.0 * (double)nM * (Md + nbnd),
           8.0 * ((double)n * MM * 2.0 + 4.0 * nM));
  TAPS_CUDA(cudaGetLastError());
  // back to the nodal basis; the previous factor goes to d_Uold
  return taps_fd_to_nodal(P, E, Y, n, M, U->d_U[d], P->d_Uold);
}
