// fr_mlp.cu -- the learned cost model of the tuner: a 16-64-64-1 ReLU MLP in
// FP32 with hand-written forward, backward (mean-squared error) and Adam
// kernels, its on-GPU training loop, and the model-ranked search order.
//
// Parameter vector (5313 floats): W1[64][16], b1[64], W2[64][64], b2[64],
// W3[64], b3 -- W[out][in].
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <numeric>
#include <random>
#include <vector>

#include "fr_ctx.h"
#include "fr_internal.h"
#include "fr_tuner.h"

namespace fr {

constexpr int OFF_W1 = 0;
constexpr int OFF_B1 = OFF_W1 + MLP_H * MLP_IN;
constexpr int OFF_W2 = OFF_B1 + MLP_H;
constexpr int OFF_B2 = OFF_W2 + MLP_H * MLP_H;
constexpr int OFF_W3 = OFF_B2 + MLP_H;
constexpr int OFF_B3 = OFF_W3 + MLP_H;
static_assert(OFF_B3 + 1 == MLP_NPARAM, "parameter layout");

// Forward and backward: CTAs of 256 threads, thread (j, q) = (tid & 63, tid >> 6)
// being hidden unit j for every fourth row of a tile of at most ROWS rows.  The
// layers are latency bound (a few microseconds of arithmetic on 152 SMs), so the
// rows are spread over all SMs (at least ROWS_MIN a tile), a unit's weights sit in
// registers (rows of W2 for the forward pass, columns for the deltas: read at
// every step from shared memory, unpadded, they cost a 32-way bank conflict),
// and the activations are read as broadcast 16-byte groups.  2970 rows: forward
// 41 -> 7 us, backward with its reduction 76 -> 21 us (cold caches; its row
// loops unrolled by four it took 24).
constexpr int ROWS = 32, ROWS_MIN = 4, MLP_T = 256, MLP_Q = MLP_T / MLP_H;
constexpr int MLP_GRID = 304;  // CTAs of a backward launch at most (partial gradients kept per CTA)

struct MlpTile {
  __align__(16) float x[ROWS][MLP_IN];
  __align__(16) float h1[ROWS][MLP_H];
  __align__(16) float h2[ROWS][MLP_H];
  __align__(16) float d2[ROWS][MLP_H];  // dL/dz2
  __align__(16) float d1[ROWS][MLP_H];  // dL/dz1
  float w1[MLP_H][MLP_IN + 1];  // padded: a row or a column per lane without bank conflicts
  float w2[MLP_H][MLP_H + 1];
  float w3[MLP_H];
  float y[ROWS];
  float dy[ROWS];
};

// rows of a tile: as few as spread m rows over the SMs
static int mlp_rows(int m) {
  const int r = (m + device_sm_count() - 1) / device_sm_count();
  return r < ROWS_MIN ? ROWS_MIN : r > ROWS ? ROWS : r;
}
static int mlp_grid(int m) {
  const int tiles = (m + mlp_rows(m) - 1) / mlp_rows(m);
  return tiles < MLP_GRID ? tiles : MLP_GRID;
}

// f(r, b + sum_k w[k] v[r][k]) for the thread's rows r = q, q + 4, ... < nrows, k
// ascending, four rows at a time: four independent chains of FMAs (v's rows are
// 16-byte aligned and read by broadcast)
template <int N, class F>
__device__ __forceinline__ void mlp_dots(const float (&w)[N], const float (*v)[N], float b, int q,
                                         int nrows, F f) {
  for (int r = q; r < nrows; r += 4 * MLP_Q) {
    float z[4] = {b, b, b, b};
#pragma unroll
    for (int k = 0; k < N; k += 4)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int ri = min(r + i * MLP_Q, nrows - 1);
        const float4 u = *reinterpret_cast<const float4 *>(v[ri] + k);
        z[i] = fmaf(w[k], u.x, z[i]);
        z[i] = fmaf(w[k + 1], u.y, z[i]);
        z[i] = fmaf(w[k + 2], u.z, z[i]);
        z[i] = fmaf(w[k + 3], u.w, z[i]);
      }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (r + i * MLP_Q < nrows) f(r + i * MLP_Q, z[i]);
  }
}

// activations and outputs of one tile's nrows rows; w1, w2: rows j of W1, W2
__device__ __forceinline__ void mlp_tile_forward(MlpTile &s, const float (&w1)[MLP_IN], float b1,
                                                 const float (&w2)[MLP_H], float b2, float b3,
                                                 const float *X, int r0, int nrows) {
  const int tid = threadIdx.x, j = tid & (MLP_H - 1), q = tid / MLP_H;
  for (int i = tid; i < nrows * MLP_IN; i += MLP_T) (&s.x[0][0])[i] = X[(size_t)r0 * MLP_IN + i];
  __syncthreads();
  mlp_dots(w1, s.x, b1, q, nrows, [&](int r, float z) { s.h1[r][j] = fmaxf(z, 0.f); });
  __syncthreads();
  mlp_dots(w2, s.h1, b2, q, nrows, [&](int r, float z) { s.h2[r][j] = fmaxf(z, 0.f); });
  __syncthreads();
  // output layer: eight lanes a row
  const int r = tid / 8, c = tid & 7;
  float z = 0.f;
  if (r < nrows)
#pragma unroll
    for (int k = 0; k < 8; ++k) z = fmaf(s.w3[c + 8 * k], s.h2[r][c + 8 * k], z);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) z += __shfl_down_sync(0xffffffffu, z, o, 8);
  if (r < nrows && c == 0) s.y[r] = z + b3;
  __syncthreads();
}

__device__ __forceinline__ void mlp_weights(const float *P, float (&w1)[MLP_IN], float &b1,
                                            float (&w2)[MLP_H], float &b2, float &b3, MlpTile &s) {
  const int j = threadIdx.x & (MLP_H - 1);
  // every load in flight before the first store (one after the other: 8 us)
  constexpr int L1 = MLP_H * MLP_IN / MLP_T, L2 = MLP_H * MLP_H / MLP_T;
  float t1[L1], t2[L2];
#pragma unroll
  for (int k = 0; k < L1; ++k) t1[k] = __ldg(P + OFF_W1 + k * MLP_T + threadIdx.x);
#pragma unroll
  for (int k = 0; k < L2; ++k) t2[k] = __ldg(P + OFF_W2 + k * MLP_T + threadIdx.x);
  b1 = __ldg(P + OFF_B1 + j);
  b2 = __ldg(P + OFF_B2 + j);
  b3 = __ldg(P + OFF_B3);
  if (threadIdx.x < MLP_H) s.w3[j] = __ldg(P + OFF_W3 + j);
#pragma unroll
  for (int k = 0; k < L1; ++k) {
    const int i = k * MLP_T + threadIdx.x;
    s.w1[i / MLP_IN][i % MLP_IN] = t1[k];
  }
#pragma unroll
  for (int k = 0; k < L2; ++k) {
    const int i = k * MLP_T + threadIdx.x;
    s.w2[i / MLP_H][i % MLP_H] = t2[k];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < MLP_IN; ++k) w1[k] = s.w1[j][k];
#pragma unroll
  for (int k = 0; k < MLP_H; ++k) w2[k] = s.w2[j][k];
}

__global__ void __launch_bounds__(MLP_T) mlp_forward_kernel(const float *P, const float *X, int m,
                                                            int rows, float *Y) {
  extern __shared__ __align__(16) unsigned char raw[];
  MlpTile &s = *reinterpret_cast<MlpTile *>(raw);
  float w1[MLP_IN], w2[MLP_H], b1, b2, b3;
  mlp_weights(P, w1, b1, w2, b2, b3, s);
  const int r0 = blockIdx.x * rows, nrows = min(rows, m - r0);
  mlp_tile_forward(s, w1, b1, w2, b2, b3, X, r0, nrows);
  if ((int)threadIdx.x < nrows) Y[r0 + threadIdx.x] = s.y[threadIdx.x];
}

// Partial gradient (and partial loss) of L = (1/m) sum (y - t)^2 over the CTA's
// tiles blockIdx.x, blockIdx.x + gridDim.x, ... into work[blockIdx.x][MLP_NPARAM
// + 1]; summed in fixed order by mlp_reduce_kernel.  Thread (j, q) holds the
// gradients of W2[j][16 q ..], W1[j][4 q ..] and, for q = 0, of unit j's biases
// and W3[j].
__global__ void __launch_bounds__(MLP_T) mlp_backward_kernel(const float *P, const float *X,
                                                             const float *T, int m, int rows,
                                                             float *work) {
  extern __shared__ __align__(16) unsigned char raw[];
  MlpTile &s = *reinterpret_cast<MlpTile *>(raw);
  const int tid = threadIdx.x, j = tid & (MLP_H - 1), q = tid / MLP_H;
  float w1[MLP_IN], w2[MLP_H], b1, b2, b3;
  mlp_weights(P, w1, b1, w2, b2, b3, s);
  float c2[MLP_H];  // column j of W2
#pragma unroll
  for (int k = 0; k < MLP_H; ++k) c2[k] = s.w2[k][j];
  constexpr int N2 = MLP_H / MLP_Q, N1 = MLP_IN / MLP_Q;
  float g2[N2] = {}, g1[N1] = {}, gb1 = 0.f, gb2 = 0.f, gw3 = 0.f, gb3 = 0.f, loss = 0.f;
  const float inv_m = 1.0f / (float)m;
  for (long long first = (long long)blockIdx.x * rows; first < m; first += (long long)gridDim.x * rows) {
    const int r0 = (int)first, nrows = min(rows, m - r0);
    mlp_tile_forward(s, w1, b1, w2, b2, b3, X, r0, nrows);
    if (tid < nrows) {
      const float e = s.y[tid] - T[r0 + tid];
      s.dy[tid] = 2.f * e * inv_m;
      s.y[tid] = e * e * inv_m;  // the row's loss term
    }
    __syncthreads();
    const float w3 = s.w3[j];
    for (int r = q; r < nrows; r += MLP_Q) s.d2[r][j] = s.h2[r][j] > 0.f ? s.dy[r] * w3 : 0.f;
    __syncthreads();
    // dW2[j][k] = sum_r d2[r][j] h1[r][k]; dz1[r][k] = [h1 > 0] sum_o W2[o][k] d2[r][o]
    for (int r = 0; r < nrows; ++r) {
      const float d = s.d2[r][j];
      const float *h = s.h1[r] + q * N2;
#pragma unroll
      for (int k = 0; k < N2; k += 4) {
        const float4 u = *reinterpret_cast<const float4 *>(h + k);
        g2[k] = fmaf(d, u.x, g2[k]);
        g2[k + 1] = fmaf(d, u.y, g2[k + 1]);
        g2[k + 2] = fmaf(d, u.z, g2[k + 2]);
        g2[k + 3] = fmaf(d, u.w, g2[k + 3]);
      }
      if (q == 0) {
        gb2 += d;
        gw3 = fmaf(s.dy[r], s.h2[r][j], gw3);
      }
    }
    mlp_dots(c2, s.d2, 0.f, q, nrows,
             [&](int r, float z) { s.d1[r][j] = s.h1[r][j] > 0.f ? z : 0.f; });
    if (tid == MLP_T - 1)
      for (int r = 0; r < nrows; ++r) {
        gb3 += s.dy[r];
        loss += s.y[r];
      }
    __syncthreads();
    for (int r = 0; r < nrows; ++r) {
      const float d = s.d1[r][j];
      const float4 u = *reinterpret_cast<const float4 *>(s.x[r] + q * N1);
      g1[0] = fmaf(d, u.x, g1[0]);
      g1[1] = fmaf(d, u.y, g1[1]);
      g1[2] = fmaf(d, u.z, g1[2]);
      g1[3] = fmaf(d, u.w, g1[3]);
      if (q == 0) gb1 += d;
    }
    __syncthreads();  // the tile is refilled
  }
  static_assert(N1 == 4 && N2 % 4 == 0, "four thread groups");
  float *G = work + (size_t)blockIdx.x * (MLP_NPARAM + 1);
#pragma unroll
  for (int k = 0; k < N2; ++k) G[OFF_W2 + j * MLP_H + q * N2 + k] = g2[k];
#pragma unroll
  for (int k = 0; k < N1; ++k) G[OFF_W1 + j * MLP_IN + q * N1 + k] = g1[k];
  if (q == 0) {
    G[OFF_B1 + j] = gb1;
    G[OFF_B2 + j] = gb2;
    G[OFF_W3 + j] = gw3;
  }
  if (tid == MLP_T - 1) {
    G[OFF_B3] = gb3;
    G[MLP_NPARAM] = loss;
  }
}

// Sum the CTAs' partial gradients: eight groups of CTAs a parameter, then the
// groups in order (fixed order: deterministic).
__global__ void __launch_bounds__(256) mlp_reduce_kernel(const float *work, int nblk, float *grad,
                                                         float *loss) {
  __shared__ float part[8][32];
  const int c = threadIdx.x & 31, gq = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + c;
  float s = 0.f;
  if (i <= MLP_NPARAM)
#pragma unroll 8
    for (int b = gq; b < nblk; b += 8) s += work[(size_t)b * (MLP_NPARAM + 1) + i];
  part[gq][c] = s;
  __syncthreads();
  if (gq == 0 && i <= MLP_NPARAM) {
    for (int k = 1; k < 8; ++k) s += part[k][c];
    if (i < MLP_NPARAM) grad[i] = s;
    else if (loss) *loss = s;
  }
}

__global__ void mlp_adam_kernel(float *P, const float *G, float *M1, float *M2, float lr, float b1,
                                float b2, float eps, float c1, float c2) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= MLP_NPARAM) return;
  float g = G[i];
  float m1 = fmaf(b1, M1[i], (1.f - b1) * g);
  float m2 = fmaf(b2, M2[i], (1.f - b2) * g * g);
  M1[i] = m1;
  M2[i] = m2;
  float mh = m1 / c1, vh = m2 / c2;
  P[i] -= lr * mh / (sqrtf(vh) + eps);
}

static bool set_attrs() {
  return allow_dynamic_smem((const void *)mlp_forward_kernel, sizeof(MlpTile)) == cudaSuccess &&
         allow_dynamic_smem((const void *)mlp_backward_kernel, sizeof(MlpTile)) == cudaSuccess;
}

size_t mlp_work_floats(int m) { return (size_t)mlp_grid(m) * (MLP_NPARAM + 1); }

cudaError_t mlp_forward(const float *params, const float *x, int m, float *y, cudaStream_t st) {
  if (m <= 0) return cudaSuccess;
  if (!set_attrs()) return cudaGetLastError();
  const int rows = mlp_rows(m);
  mlp_forward_kernel<<<(m + rows - 1) / rows, MLP_T, sizeof(MlpTile), st>>>(params, x, m, rows, y);
  return cudaGetLastError();
}

cudaError_t mlp_backward(const float *params, const float *x, const float *t, int m, float *grad,
                         float *loss, float *work, cudaStream_t st) {
  if (m <= 0) return cudaErrorInvalidValue;
  if (!set_attrs()) return cudaGetLastError();
  const int nblk = mlp_grid(m);
  mlp_backward_kernel<<<nblk, MLP_T, sizeof(MlpTile), st>>>(params, x, t, m, mlp_rows(m), work);
  mlp_reduce_kernel<<<(MLP_NPARAM + 1 + 31) / 32, 256, 0, st>>>(work, nblk, grad, loss);
  return cudaGetLastError();
}

cudaError_t mlp_adam(float *params, const float *grad, float *m1, float *m2, int t, float lr,
                     float b1, float b2, float eps, cudaStream_t st) {
  float c1 = 1.f - std::pow(b1, (float)t), c2 = 1.f - std::pow(b2, (float)t);
  mlp_adam_kernel<<<(MLP_NPARAM + 255) / 256, 256, 0, st>>>(params, grad, m1, m2, lr, b1, b2, eps,
                                                            c1, c2);
  return cudaGetLastError();
}

// Stream-ordered workspace of fr_mlp_backward, from a pool per device that keeps
// up to WORK_KEEP bytes between calls (a gradient's partial sums are at most 6.5
// MB): the default pool hands its memory back at every synchronisation, and a call
// that follows one waited 170 us for new memory.
static cudaError_t work_alloc(float **p, size_t bytes, cudaStream_t st) {
  constexpr unsigned long long WORK_KEEP = 8ull << 20;
  static std::mutex mu;
  static std::vector<cudaMemPool_t> pools;  // by device ordinal
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  cudaMemPool_t pool = nullptr;
  {
    std::lock_guard<std::mutex> lk(mu);
    if ((int)pools.size() <= dev) pools.resize(dev + 1, nullptr);
    if (!pools[dev]) {
      cudaMemPoolProps props{};
      props.allocType = cudaMemAllocationTypePinned;
      props.location.type = cudaMemLocationTypeDevice;
      props.location.id = dev;
      unsigned long long keep = WORK_KEEP;
      if (cudaMemPoolCreate(&pools[dev], &props) != cudaSuccess ||
          cudaMemPoolSetAttribute(pools[dev], cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
        cudaGetLastError();
        pools[dev] = nullptr;
      }
    }
    pool = pools[dev];
  }
  void *q = nullptr;
  e = pool ? cudaMallocFromPoolAsync(&q, bytes, pool, st) : cudaMallocAsync(&q, bytes, st);
  *p = static_cast<float *>(q);
  return e;
}

// He-uniform initialisation on the host from a seed.
static void init_params(std::vector<float> &p, unsigned long long seed) {
  std::mt19937_64 rng(seed);
  p.assign(MLP_NPARAM, 0.f);
  auto fill = [&](int off, int nout, int nin) {
    float lim = std::sqrt(6.f / (float)nin);
    std::uniform_real_distribution<float> u(-lim, lim);
    for (int i = 0; i < nout * nin; ++i) p[off + i] = u(rng);
  };
  fill(OFF_W1, MLP_H, MLP_IN);
  fill(OFF_W2, MLP_H, MLP_H);
  fill(OFF_W3, 1, MLP_H);
}

// Model-ranked search order: predicted time ascending, ties by configuration id.
std::vector<int> learned_order(fr_ctx *c, const TuneKey &k, const std::vector<int> &valid,
                               int *predicted_best) {
  std::vector<int> order = valid;
  const int m = (int)valid.size();
  if (m == 0 || !c->d_mlp) return order;
  std::vector<float> feat((size_t)m * MLP_IN), pred(m);
  const int n_repr = (int)std::min<long long>(1LL << 24, (3LL << k.nb) / 2);  // bucket middle
  for (int i = 0; i < m; ++i)
    config_features(effective_config(valid[i], k.S, k.a), k.S, n_repr, k.a, &feat[(size_t)i * MLP_IN]);
  float *dx = nullptr, *dy = nullptr;
  if (cudaMalloc(&dx, feat.size() * sizeof(float)) != cudaSuccess) return order;
  if (cudaMalloc(&dy, m * sizeof(float)) != cudaSuccess) { cudaFree(dx); return order; }
  cudaMemcpy(dx, feat.data(), feat.size() * sizeof(float), cudaMemcpyHostToDevice);
  mlp_forward(c->d_mlp, dx, m, dy, 0);
  cudaMemcpy(pred.data(), dy, m * sizeof(float), cudaMemcpyDeviceToHost);
  cudaFree(dx);
  cudaFree(dy);
  std::vector<int> idx(m);
  std::iota(idx.begin(), idx.end(), 0);
  std::stable_sort(idx.begin(), idx.end(), [&](int a, int b) {
    if (pred[a] != pred[b]) return pred[a] < pred[b];
    return valid[a] < valid[b];
  });
  for (int i = 0; i < m; ++i) order[i] = valid[idx[i]];
  if (predicted_best) *predicted_best = order[0];
  return order;
}

}  // namespace fr

using namespace fr;

extern "C" {

int fr_mlp_num_params(void) { return MLP_NPARAM; }

int fr_mlp_forward(const float *params, const float *x, int m, float *y, void *stream) {
  if (m < 0 || (m > 0 && (!params || !x || !y))) return FR_ERR_INVALID_ARG;
  return mlp_forward(params, x, m, y, (cudaStream_t)stream) == cudaSuccess ? FR_OK : FR_ERR_CUDA;
}

int fr_mlp_backward(const float *params, const float *x, const float *target, int m, float *grad,
                    float *loss, void *stream) {
  if (m < 1 || !params || !x || !target || !grad || !loss) return FR_ERR_INVALID_ARG;
  float *work = nullptr;
  if (work_alloc(&work, mlp_work_floats(m) * sizeof(float), (cudaStream_t)stream) != cudaSuccess)
    return FR_ERR_OOM;
  cudaError_t e = mlp_backward(params, x, target, m, grad, loss, work, (cudaStream_t)stream);
  cudaFreeAsync(work, (cudaStream_t)stream);
  return e == cudaSuccess ? FR_OK : FR_ERR_CUDA;
}

int fr_mlp_adam(float *params, const float *grad, float *m1, float *m2, int t, float lr,
                float beta1, float beta2, float eps, void *stream) {
  if (!params || !grad || !m1 || !m2 || t < 1) return FR_ERR_INVALID_ARG;
  return mlp_adam(params, grad, m1, m2, t, lr, beta1, beta2, eps, (cudaStream_t)stream) ==
                 cudaSuccess
             ? FR_OK
             : FR_ERR_CUDA;
}

int fr_mlp_train(fr_ctx *c, const float *feat, const float *logt, int m, int epochs, float lr,
                 uint64_t seed, float *final_loss) {
  if (!c || !feat || !logt || m < 1 || epochs < 0) return FR_ERR_INVALID_ARG;
  std::vector<float> p;
  init_params(p, seed);
  if (!c->d_mlp && cudaMalloc(&c->d_mlp, MLP_NPARAM * sizeof(float)) != cudaSuccess)
    return FR_ERR_OOM;
  float *X = nullptr, *T = nullptr, *G = nullptr, *M1 = nullptr, *M2 = nullptr, *W = nullptr,
        *L = nullptr;
  size_t wn = mlp_work_floats(m);
  bool ok = cudaMalloc(&X, (size_t)m * MLP_IN * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&T, (size_t)m * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&G, MLP_NPARAM * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&M1, MLP_NPARAM * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&M2, MLP_NPARAM * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&W, wn * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&L, sizeof(float)) == cudaSuccess;
  int rc = FR_OK;
  if (!ok) rc = FR_ERR_OOM;
  if (rc == FR_OK) {
    cudaMemcpy(c->d_mlp, p.data(), MLP_NPARAM * sizeof(float), cudaMemcpyHostToDevice);
    cudaMemcpy(X, feat, (size_t)m * MLP_IN * sizeof(float), cudaMemcpyHostToDevice);
    cudaMemcpy(T, logt, (size_t)m * sizeof(float), cudaMemcpyHostToDevice);
    cudaMemset(M1, 0, MLP_NPARAM * sizeof(float));
    cudaMemset(M2, 0, MLP_NPARAM * sizeof(float));
    cudaMemset(L, 0, sizeof(float));
    for (int t = 1; t <= epochs; ++t) {
      if (mlp_backward(c->d_mlp, X, T, m, G, L, W, 0) != cudaSuccess ||
          mlp_adam(c->d_mlp, G, M1, M2, t, lr, 0.9f, 0.999f, 1e-8f, 0) != cudaSuccess) {
        rc = FR_ERR_CUDA;
        break;
      }
    }
    if (rc == FR_OK) {
      // loss of the final parameters
      if (mlp_backward(c->d_mlp, X, T, m, G, L, W, 0) != cudaSuccess) rc = FR_ERR_CUDA;
      float l = 0.f;
      if (cudaMemcpy(&l, L, sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess) rc = FR_ERR_CUDA;
      if (final_loss) *final_loss = l;
    }
  }
  cudaFree(X); cudaFree(T); cudaFree(G); cudaFree(M1); cudaFree(M2); cudaFree(W); cudaFree(L);
  if (rc == FR_OK) {
    c->mlp_trained = true;
    c->tuner.retune(true);
  }
  return rc;
}

int fr_mlp_get(const fr_ctx *c, float *params_host) {
  if (!c || !params_host) return FR_ERR_INVALID_ARG;
  if (!c->d_mlp) return FR_ERR_STATE;
  return cudaMemcpy(params_host, c->d_mlp, MLP_NPARAM * sizeof(float), cudaMemcpyDeviceToHost) ==
                 cudaSuccess
             ? FR_OK
             : FR_ERR_CUDA;
}

int fr_mlp_set(fr_ctx *c, const float *params_host) {
  if (!c || !params_host) return FR_ERR_INVALID_ARG;
  if (!c->d_mlp && cudaMalloc(&c->d_mlp, MLP_NPARAM * sizeof(float)) != cudaSuccess)
    return FR_ERR_OOM;
  if (cudaMemcpy(c->d_mlp, params_host, MLP_NPARAM * sizeof(float), cudaMemcpyHostToDevice) !=
      cudaSuccess)
    return FR_ERR_CUDA;
  c->mlp_trained = true;
  c->tuner.retune(true);
  return FR_OK;
}

}  // extern "C"
