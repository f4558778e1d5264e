// Learned warm start: a fully connected network (FP32) that maps an instance's
// parameter vector and a mode index to initial factor profiles, with hand-written
// forward, backward and Adam kernels, and the kernel that turns predicted profiles
// into initial factor columns (the paper's Algorithm 1 starts from random values;
// this replaces them by a learned proposal).
//
// Network: n_in -> H -> ... -> H -> n_out, tanh after every hidden layer, linear
// output; loss = mean squared error over the batch and outputs.  Parameters are one
// flat FP32 array: for each layer l, W_l [out][in] row-major, then b_l [out].
#include <string.h>

#include <algorithm>

#include "taps_internal.cuh"

struct taps_mlp {
  int L;                      // linear layers
  int dims[TAPS_MLP_MAX_LAYERS + 1];
  size_t woff[TAPS_MLP_MAX_LAYERS], boff[TAPS_MLP_MAX_LAYERS];
  size_t nparams;
  float *d_p, *d_g, *d_m, *d_v;  // parameters, gradients, Adam moments
  long long t;                   // Adam step count
  cudaStream_t stream;
  int cap;                       // batch capacity of the activation buffers
  float* d_act;                  // activations A_0 .. A_L, [cap][dims[l]] each
  float* d_dact;                 // gradient buffers, same layout
  size_t aoff[TAPS_MLP_MAX_LAYERS + 1];
  float* d_loss;                 // per-block loss partials
  float* h_loss;
  int* d_status;
};

// ---------------------------------------------------------------------------------
// C[r][c] = sum_k X(r,k) Y(k,c), X(r,k) = X[r*sxr + k*sxk], Y(k,c) = Y[k*syk + c*syc], C
// row-major with leading dimension ldc, and an epilogue (see MlpJob).  A launch holds one
// product or two independent ones (a layer's dA and dW), tiles of the second after the first's.
//
// The products of this network are small (480 x 256 x 256: 0.9 us of FP32 at the chip's
// rate), so a launch is latency: 32 x 32 tiles put 120 CTAs on the GPU, and the next 64-wide
// k slice is loaded to registers while the current one is multiplied.  Two by four outputs to
// a thread: the shared-memory reads are the bound (an LDS.128 takes four cycles whatever it
// broadcasts), one by four was 1.5 times slower.  480 x 256 x 256: 22 us per launch with one
// output column per thread and no prefetch, 8.7 us now; four groups of warps sharing out k
// would be faster still, but re-rounds every training run.  Operands lie [k][row] in shared
// memory whatever their strides.  Each output is one FMA chain in increasing k, as
// are the bias gradients, so results depend neither on the tiling nor on the batch.
// ---------------------------------------------------------------------------------
#define MT 32           // tile edge
#define MLP_THREADS 128
#define MLP_BK 64       // k slice
#define MLP_FRAG 4      // k's per register fragment
#define MLP_LD 36       // row stride of a k slice: 16-byte aligned rows
#define MLP_SLICE ((MLP_BK + MLP_FRAG) * MLP_LD)   // a slice and the fragment read ahead of its end
enum { MLP_PLAIN, MLP_TANH, MLP_OUT, MLP_TANH_BACK };
struct MlpJob {
  const float *X, *Y;
  long long sxr, sxk, syk, syc;
  int xk, yk;            // unit stride along k
  float* C;
  int ldc, R, Cn, K;
  int epi;               // MLP_TANH: + bias, tanh; MLP_OUT: + bias, and dY below; MLP_TANH_BACK: * (1 - aux^2)
  const float* bias;
  const float* aux;      // MLP_OUT: targets (or null); MLP_TANH_BACK: the layer's activations; as C
  float* dY;             // MLP_OUT: 2 (C - target) scale
  float scale;
  float* db;             // bias gradient sum_k X(r, k) (or null), by the tiles of the first column
  int tiles_x, tiles;
};
struct MlpJobs {
  MlpJob j[2];
};

// The elements of one operand's k slices that a thread carries from global to shared memory.
// ALONG_K (unit stride along k): eight k by four rows to a warp, whole 32-byte sectors in
// global memory and no bank conflicts in the transposing store; else 32 rows by one k.
template <bool ALONG_K>
struct MlpSlice {
  static constexpr int PER = MT * MLP_BK / MLP_THREADS;
  const float* p;        // element 0 of the next slice
  long long jump;        // ALONG_K: 16 rows, else 4 k
  long long slice;       // MLP_BK k
  int k, r, rows;        // element 0 in the slice; rows of the operand from the tile's first
  float v[PER];
  __device__ __forceinline__ MlpSlice(const float* base, long long sr, long long sk, int row0, int nrows) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    k = ALONG_K ? lane & 7 : w;
    r = ALONG_K ? (lane >> 3) + 4 * w : lane;
    rows = nrows - row0;
    jump = ALONG_K ? 16 * sr : 4 * sk;
    slice = MLP_BK * sk;
    p = base + (row0 + r) * sr + k * sk;
  }
  __device__ __forceinline__ void fetch(int left) {   // left: k's from the slice's first on
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int kk = ALONG_K ? k + 8 * (q & 7) : k + 4 * q;
      const bool in = kk < left && (ALONG_K ? r + 16 * (q >> 3) : r) < rows;
      v[q] = in ? __ldg(ALONG_K ? p + (q >> 3) * jump + 8 * (q & 7) : p + q * jump) : 0.f;
    }
    p += slice;
  }
  __device__ __forceinline__ void store(float* s) const {
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int kk = ALONG_K ? k + 8 * (q & 7) : k + 4 * q;
      s[kk * MLP_LD + (ALONG_K ? r + 16 * (q >> 3) : r)] = v[q];
    }
  }
};

template <bool XK, bool YK>
__device__ __forceinline__ void mlp_tile(const MlpJob& job, int tile, float (*Xs)[MLP_SLICE], float (*Ys)[MLP_SLICE]) {
  const MlpJob J = job;
  const int r0 = tile / J.tiles_x * MT, c0 = tile % J.tiles_x * MT;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  MlpSlice<XK> X(J.X, J.sxr, J.sxk, r0, J.R);
  MlpSlice<YK> Y(J.Y, J.syc, J.syk, c0, J.Cn);
  const int nk = (J.K + MLP_BK - 1) / MLP_BK;
  X.fetch(J.K);
  Y.fetch(J.K);
  X.store(Xs[0]);
  Y.store(Ys[0]);
  __syncthreads();
  const int tx = tid & 7, ty = tid >> 3;   // columns 4 tx .., rows 2 ty ..
  float acc[2][4] = {};
  float bsum = 0.f;
  const bool bias_sum = J.db && c0 == 0 && w == 0;
  for (int t = 0; t < nk; ++t) {
    if (t + 1 < nk) {
      X.fetch(J.K - (t + 1) * MLP_BK);
      Y.fetch(J.K - (t + 1) * MLP_BK);
    }
    const float* xs = Xs[t & 1] + 2 * ty;
    const float* ys = Ys[t & 1] + 4 * tx;
    // fragments four k ahead of the FMAs hide the shared-memory latency
    float2 x[2][MLP_FRAG];
    float4 y[2][MLP_FRAG];
#pragma unroll
    for (int i = 0; i < MLP_FRAG; ++i) {
      x[0][i] = *reinterpret_cast<const float2*>(xs + i * MLP_LD);
      y[0][i] = *reinterpret_cast<const float4*>(ys + i * MLP_LD);
    }
#pragma unroll 2
    for (int k = 0; k < MLP_BK; k += 2 * MLP_FRAG) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int kn = k + (h + 1) * MLP_FRAG;   // rows past the slice are the pad's
#pragma unroll
        for (int i = 0; i < MLP_FRAG; ++i) {
          x[h ^ 1][i] = *reinterpret_cast<const float2*>(xs + (kn + i) * MLP_LD);
          y[h ^ 1][i] = *reinterpret_cast<const float4*>(ys + (kn + i) * MLP_LD);
        }
#pragma unroll
        for (int i = 0; i < MLP_FRAG; ++i) {
          const float2 u = x[h][i];
          const float4 v = y[h][i];
          acc[0][0] = fmaf(u.x, v.x, acc[0][0]);
          acc[0][1] = fmaf(u.x, v.y, acc[0][1]);
          acc[0][2] = fmaf(u.x, v.z, acc[0][2]);
          acc[0][3] = fmaf(u.x, v.w, acc[0][3]);
          acc[1][0] = fmaf(u.y, v.x, acc[1][0]);
          acc[1][1] = fmaf(u.y, v.y, acc[1][1]);
          acc[1][2] = fmaf(u.y, v.z, acc[1][2]);
          acc[1][3] = fmaf(u.y, v.w, acc[1][3]);
        }
      }
    }
    if (bias_sum)
#pragma unroll 16
      for (int k = 0; k < MLP_BK; ++k) bsum += Xs[t & 1][k * MLP_LD + lane];
    if (t + 1 < nk) {   // the other buffer was read last in slice t - 1, before the last barrier
      X.store(Xs[(t + 1) & 1]);
      Y.store(Ys[(t + 1) & 1]);
      __syncthreads();
    }
  }
  if (bias_sum && r0 + lane < J.R) J.db[r0 + lane] = bsum;
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const int r = r0 + 2 * ty + a;
    if (r >= J.R) continue;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int c = c0 + 4 * tx + b;
      if (c >= J.Cn) continue;
      const size_t at = (size_t)r * J.ldc + c;
      float v = acc[a][b] + (J.bias ? J.bias[c] : 0.f);
      if (J.epi == MLP_TANH) v = tanhf(v);
      if (J.epi == MLP_TANH_BACK) v *= 1.f - J.aux[at] * J.aux[at];
      J.C[at] = v;
      if (J.epi == MLP_OUT && J.aux) {
        const float d = v - J.aux[at];
        J.dY[at] = 2.f * d * J.scale;
      }
    }
  }
}

__global__ void __launch_bounds__(MLP_THREADS) mlp_gemm_kernel(const __grid_constant__ MlpJobs jobs) {
  __shared__ __align__(16) float Xs[2][MLP_SLICE];
  __shared__ __align__(16) float Ys[2][MLP_SLICE];
  const int second = (int)blockIdx.x >= jobs.j[0].tiles ? 1 : 0;
  const MlpJob& J = jobs.j[second];
  const int tile = blockIdx.x - (second ? jobs.j[0].tiles : 0);
  taps_pdl_wait();
  if (J.xk && J.yk) mlp_tile<true, true>(J, tile, Xs, Ys);         // forward
  else if (J.xk) mlp_tile<true, false>(J, tile, Xs, Ys);           // dA
  else mlp_tile<false, false>(J, tile, Xs, Ys);                    // dW
}

// Loss partials.
__global__ void mlp_mse_kernel(const float* __restrict__ Yp, const float* __restrict__ T, long long n,
                               float* __restrict__ partial) {
  __shared__ float red[32];
  taps_pdl_wait();
  float s = 0.f;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    float d = Yp[i] - T[i];
    s += d * d;
  }
  s = block_sum(s, red);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

// Adam with bias correction.
__global__ void mlp_adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                                float* __restrict__ v, long long n, float lr, float b1, float b2, float eps,
                                float c1, float c2) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  taps_pdl_wait();
  float gi = g[i];
  float mi = b1 * m[i] + (1.f - b1) * gi;
  float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// Xavier-uniform weights from SplitMix64 draws keyed on (seed, parameter index); zero biases.
__global__ void mlp_init_kernel(float* __restrict__ p, long long woff, long long boff, int in, int out,
                                unsigned seed) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  long long nw = (long long)in * out;
  if (i < nw) {
    double u = taps_uniform_pm1(seed, 0xEE, (int)(i & 0xFFFFF), (int)((woff + (i >> 20)) & 0xFFF));
    float lim = sqrtf(6.f / (float)(in + out));
    p[woff + i] = (float)u * lim;
  } else if (i < nw + out) {
    p[boff + (i - nw)] = 0.f;
  }
}

// ---------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------
static MlpJob job(const float* X, long long sxr, long long sxk, const float* Y, long long syk, long long syc, float* C,
                  int ldc, int R, int Cn, int K, int epi) {
  MlpJob J;
  memset(&J, 0, sizeof(J));
  J.X = X;
  J.sxr = sxr;
  J.sxk = sxk;
  J.Y = Y;
  J.syk = syk;
  J.syc = syc;
  J.C = C;
  J.ldc = ldc;
  J.R = R;
  J.Cn = Cn;
  J.K = K;
  J.epi = epi;
  J.xk = epi != MLP_PLAIN;   // dW = G^T A takes both operands along the batch, the others' X is row-major
  J.yk = epi == MLP_TANH || epi == MLP_OUT;   // forward: Y = W^T
  J.tiles_x = (Cn + MT - 1) / MT;
  J.tiles = J.tiles_x * ((R + MT - 1) / MT);
  return J;
}

// One product, or two that do not depend on each other.
static int gemm(cudaStream_t s, const MlpJob& a, const MlpJob* b = nullptr) {
  MlpJobs jobs;
  memset(&jobs, 0, sizeof(jobs));
  jobs.j[0] = a;
  if (b) jobs.j[1] = *b;
  TAPS_CUDA(taps_launch_pdl(mlp_gemm_kernel, dim3(a.tiles + (b ? b->tiles : 0)), dim3(MLP_THREADS), 0, s, jobs));
  return TAPS_OK;
}

static int mlp_ensure_batch(taps_mlp* N, int B) {
  if (B <= N->cap) return TAPS_OK;
  cudaFree(N->d_act);
  cudaFree(N->d_dact);
  N->d_act = N->d_dact = nullptr;
  size_t tot = 0;
  for (int l = 0; l <= N->L; ++l) {
    N->aoff[l] = tot;
    tot += (size_t)B * N->dims[l];
  }
  TAPS_TRY(taps_alloc((void**)&N->d_act, sizeof(float) * tot));
  TAPS_TRY(taps_alloc((void**)&N->d_dact, sizeof(float) * tot));
  N->cap = B;
  return TAPS_OK;
}

extern "C" void taps_mlp_destroy(taps_mlp* N) {
  if (!N) return;
  if (N->stream) cudaStreamSynchronize(N->stream);
  cudaFree(N->d_p);
  cudaFree(N->d_g);
  cudaFree(N->d_m);
  cudaFree(N->d_v);
  cudaFree(N->d_act);
  cudaFree(N->d_dact);
  cudaFree(N->d_loss);
  cudaFree(N->d_status);
  if (N->h_loss) cudaFreeHost(N->h_loss);
  delete N;
}

extern "C" int taps_mlp_create(int n_in, int n_hidden, int hidden_layers, int n_out, unsigned seed, void* stream,
                               taps_mlp** out) {
  if (!out || n_in < 1 || n_hidden < 1 || n_out < 1 || hidden_layers < 0 ||
      hidden_layers + 1 > TAPS_MLP_MAX_LAYERS)
    return TAPS_ERR_INVALID_ARG;
  *out = nullptr;
  taps_mlp* N = new taps_mlp();
  memset((void*)N, 0, sizeof(taps_mlp));
  N->L = hidden_layers + 1;
  N->dims[0] = n_in;
  for (int l = 1; l < N->L; ++l) N->dims[l] = n_hidden;
  N->dims[N->L] = n_out;
  N->stream = (cudaStream_t)stream;
  size_t off = 0;
  for (int l = 0; l < N->L; ++l) {
    N->woff[l] = off;
    off += (size_t)N->dims[l] * N->dims[l + 1];
    N->boff[l] = off;
    off += N->dims[l + 1];
  }
  N->nparams = off;
  int st = TAPS_OK;
  do {
    if ((st = taps_alloc((void**)&N->d_p, sizeof(float) * off)) != TAPS_OK) break;
    if ((st = taps_alloc((void**)&N->d_g, sizeof(float) * off)) != TAPS_OK) break;
    if ((st = taps_alloc((void**)&N->d_m, sizeof(float) * off)) != TAPS_OK) break;
    if ((st = taps_alloc((void**)&N->d_v, sizeof(float) * off)) != TAPS_OK) break;
    if ((st = taps_alloc((void**)&N->d_loss, sizeof(float) * 256)) != TAPS_OK) break;
    if ((st = taps_alloc((void**)&N->d_status, sizeof(int))) != TAPS_OK) break;
    if (cudaMallocHost((void**)&N->h_loss, sizeof(float) * 256) != cudaSuccess) { st = TAPS_ERR_OOM; break; }
    cudaMemsetAsync(N->d_m, 0, sizeof(float) * off, N->stream);
    cudaMemsetAsync(N->d_v, 0, sizeof(float) * off, N->stream);
    cudaMemsetAsync(N->d_g, 0, sizeof(float) * off, N->stream);
    for (int l = 0; l < N->L; ++l) {
      long long n = (long long)N->dims[l] * N->dims[l + 1] + N->dims[l + 1];
      mlp_init_kernel<<<(unsigned)((n + 255) / 256), 256, 0, N->stream>>>(
          N->d_p, (long long)N->woff[l], (long long)N->boff[l], N->dims[l], N->dims[l + 1], seed + 977u * l);
    }
    if (cudaGetLastError() != cudaSuccess) { st = TAPS_ERR_CUDA; break; }
    if (cudaStreamSynchronize(N->stream) != cudaSuccess) { st = TAPS_ERR_CUDA; break; }
  } while (0);
  if (st != TAPS_OK) {
    taps_mlp_destroy(N);
    return st;
  }
  *out = N;
  return TAPS_OK;
}

extern "C" long long taps_mlp_num_params(const taps_mlp* N) { return N ? (long long)N->nparams : -1; }

extern "C" int taps_mlp_get_params(const taps_mlp* N, float* host, long long n) {
  if (!N || !host || n != (long long)N->nparams) return TAPS_ERR_INVALID_ARG;
  TAPS_CUDA(cudaMemcpyAsync(host, N->d_p, sizeof(float) * n, cudaMemcpyDeviceToHost, N->stream));
  TAPS_CUDA(cudaStreamSynchronize(N->stream));
  return TAPS_OK;
}

extern "C" int taps_mlp_set_params(taps_mlp* N, const float* host, long long n) {
  if (!N || !host || n != (long long)N->nparams) return TAPS_ERR_INVALID_ARG;
  TAPS_CUDA(cudaMemcpyAsync(N->d_p, host, sizeof(float) * n, cudaMemcpyHostToDevice, N->stream));
  TAPS_CUDA(cudaStreamSynchronize(N->stream));
  N->t = 0;
  TAPS_CUDA(cudaMemsetAsync(N->d_m, 0, sizeof(float) * n, N->stream));
  TAPS_CUDA(cudaMemsetAsync(N->d_v, 0, sizeof(float) * n, N->stream));
  return TAPS_OK;
}

// Forward pass from x into the activation buffers, the output to y; with targets t also
// dY = 2 (y - t) scale.
static int mlp_forward_impl(taps_mlp* N, const float* x_dev, int B, float* y, const float* t, float* dY, float scale) {
  for (int l = 0; l < N->L; ++l) {
    const int in = N->dims[l], o = N->dims[l + 1];
    const bool last = l == N->L - 1;
    // Z[b][o] = sum_i A[b][i] W[o][i] + b[o]
    MlpJob J = job(l == 0 ? x_dev : N->d_act + N->aoff[l], in, 1, N->d_p + N->woff[l], 1, in,
                   last ? y : N->d_act + N->aoff[l + 1], o, B, o, in, last ? MLP_OUT : MLP_TANH);
    J.bias = N->d_p + N->boff[l];
    if (last) {
      J.aux = t;
      J.dY = dY;
      J.scale = scale;
    }
    TAPS_TRY(gemm(N->stream, J));
  }
  return TAPS_OK;
}

extern "C" int taps_mlp_forward(taps_mlp* N, const float* x_dev, int batch, float* y_dev) {
  if (!N || !x_dev || !y_dev || batch < 1) return TAPS_ERR_INVALID_ARG;
  TAPS_TRY(mlp_ensure_batch(N, batch));
  // a single layer reads x while it writes y: through the buffer, so that they may overlap
  float* y = N->L > 1 ? y_dev : N->d_act + N->aoff[N->L];
  TAPS_TRY(mlp_forward_impl(N, x_dev, batch, y, nullptr, nullptr, 0.f));
  if (y != y_dev)
    TAPS_CUDA(cudaMemcpyAsync(y_dev, y, sizeof(float) * batch * N->dims[N->L], cudaMemcpyDeviceToDevice, N->stream));
  return TAPS_OK;
}

// Loss and parameter gradients of one batch (gradients into the internal buffer).
static int mlp_grad_impl(taps_mlp* N, const float* x_dev, const float* t_dev, int B, int want_loss, float* loss) {
  TAPS_TRY(mlp_ensure_batch(N, B));
  cudaStream_t s = N->stream;
  const int O = N->dims[N->L];
  const long long n = (long long)B * O;
  float* y = N->d_act + N->aoff[N->L];
  TAPS_TRY(mlp_forward_impl(N, x_dev, B, y, t_dev, N->d_dact + N->aoff[N->L], 1.f / (float)n));
  for (int l = N->L - 1; l >= 0; --l) {
    const int in = N->dims[l], o = N->dims[l + 1];
    const float* A = l == 0 ? x_dev : N->d_act + N->aoff[l];
    float* Gl = N->d_dact + N->aoff[l + 1];
    // dW[o][i] = sum_b G[b][o] A[b][i], db[o] = sum_b G[b][o]
    MlpJob W = job(Gl, 1, o, A, in, 1, N->d_g + N->woff[l], in, o, in, B, MLP_PLAIN);
    W.db = N->d_g + N->boff[l];
    if (l == 0) {
      TAPS_TRY(gemm(s, W));
      break;
    }
    // dA[b][i] = sum_o G[b][o] W[o][i], times tanh' in terms of the activation A
    MlpJob D = job(Gl, o, 1, N->d_p + N->woff[l], in, 1, N->d_dact + N->aoff[l], in, B, in, o, MLP_TANH_BACK);
    D.aux = A;
    TAPS_TRY(gemm(s, D, &W));
  }
  if (want_loss) {
    TAPS_CUDA(taps_launch_pdl(mlp_mse_kernel, dim3(64), dim3(256), 0, s, (const float*)y, t_dev, n, N->d_loss));
    TAPS_CUDA(cudaMemcpyAsync(N->h_loss, N->d_loss, sizeof(float) * 64, cudaMemcpyDeviceToHost, s));
    TAPS_CUDA(cudaStreamSynchronize(s));
    double acc = 0.0;
    for (int b = 0; b < 64; ++b) acc += N->h_loss[b];
    *loss = (float)(acc / (double)n);
  }
  return TAPS_OK;
}

extern "C" int taps_mlp_grad(taps_mlp* N, const float* x_dev, const float* t_dev, int batch, float* loss_out,
                             float* grad_host) {
  if (!N || !x_dev || !t_dev || batch < 1) return TAPS_ERR_INVALID_ARG;
  float loss = 0.f;
  TAPS_TRY(mlp_grad_impl(N, x_dev, t_dev, batch, 1, &loss));
  if (loss_out) *loss_out = loss;
  if (grad_host) {
    TAPS_CUDA(cudaMemcpyAsync(grad_host, N->d_g, sizeof(float) * N->nparams, cudaMemcpyDeviceToHost, N->stream));
    TAPS_CUDA(cudaStreamSynchronize(N->stream));
  }
  return TAPS_OK;
}

extern "C" int taps_mlp_adam(taps_mlp* N, float lr, float beta1, float beta2, float eps) {
  if (!N) return TAPS_ERR_INVALID_ARG;
  N->t += 1;
  float c1 = 1.f - powf(beta1, (float)N->t), c2 = 1.f - powf(beta2, (float)N->t);
  long long n = (long long)N->nparams;
  TAPS_CUDA(taps_launch_pdl(mlp_adam_kernel, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, N->stream, N->d_p,
                            (const float*)N->d_g, N->d_m, N->d_v, n, lr, beta1, beta2, eps, c1, c2));
  return TAPS_OK;
}

extern "C" int taps_mlp_train(taps_mlp* N, const float* x_dev, const float* t_dev, int batch, int steps, float lr,
                              float* loss_out) {
  if (!N || !x_dev || !t_dev || batch < 1 || steps < 0) return TAPS_ERR_INVALID_ARG;
  float loss = 0.f;
  for (int it = 0; it < steps; ++it) {
    TAPS_TRY(mlp_grad_impl(N, x_dev, t_dev, batch, it == steps - 1, &loss));
    TAPS_TRY(taps_mlp_adam(N, lr, 0.9f, 0.999f, 1e-8f));
  }
  TAPS_CUDA(cudaStreamSynchronize(N->stream));
  if (loss_out) *loss_out = loss;
  return TAPS_OK;
}

// ---------------------------------------------------------------------------------
// Predicted profiles -> initial factors.  prof is [M][D * n_ref + 1] (FP32): per dim a
// profile sampled at n_ref uniform points of [lo_d, hi_d], then the mode weight.
// U_d[j, m] = linear interpolation of the profile at the free node j; the weight
// multiplies the last dim.
// ---------------------------------------------------------------------------------
struct ProfileDims {
  int nf[TAPS_MAX_DIMS], off[TAPS_MAX_DIMS], n[TAPS_MAX_DIMS];
  double* U[TAPS_MAX_DIMS];
};

__global__ void profiles_to_factors_kernel(const float* __restrict__ prof, ProfileDims pd, int D, int M, int n_ref,
                                           int d, double wscale) {
  int idx = blockIdx.x * blockDim.x + threadIdx.x;
  int nf = pd.nf[d];
  if (idx >= nf * M) return;
  int m = idx / nf, j = idx % nf;
  int node = j + pd.off[d];
  double t = (double)node / (double)(pd.n[d] - 1) * (double)(n_ref - 1);
  int k = min((int)floor(t), n_ref - 2);
  double f = t - k;
  const float* p = prof + (size_t)m * (D * n_ref + 1) + (size_t)d * n_ref;
  double v = (1.0 - f) * (double)p[k] + f * (double)p[k + 1];
  if (d == D - 1) v *= wscale * (double)prof[(size_t)m * (D * n_ref + 1) + D * n_ref];
  pd.U[d][(size_t)m * nf + j] = v;
}

extern "C" int taps_factors_from_profiles(const taps_problem* P, taps_factors* U, int M, const float* prof_dev,
                                          int n_ref, double weight_scale) {
  if (!P || !U || !prof_dev || M < 1 || M > U->M_cap || n_ref < 2) return TAPS_ERR_INVALID_ARG;
  ProfileDims pd;
  memset(&pd, 0, sizeof(pd));
  for (int d = 0; d < P->D; ++d) {
    pd.nf[d] = P->dims[d]->nf;
    pd.off[d] = P->dims[d]->off;
    pd.n[d] = P->dims[d]->n;
    pd.U[d] = U->d_U[d];
  }
  for (int d = 0; d < P->D; ++d) {
    int n = pd.nf[d] * M;
    profiles_to_factors_kernel<<<(n + 255) / 256, 256, 0, P->stream>>>(prof_dev, pd, P->D, M, n_ref, d,
                                                                        weight_scale);
  }
  TAPS_CUDA(cudaGetLastError());
  TAPS_CUDA(cudaStreamSynchronize(P->stream));
  U->M = M;
  return TAPS_OK;
}
