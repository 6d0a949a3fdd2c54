// k_mlp.cu -- the learned tile-cost model: a 16 -> 128 -> 128 -> 1 MLP with
// exact GELU, trained with MSE and Adam, all on the GPU in FP32.
//
// It ranks candidate tile schedules (tile sizes, stages, cluster, split-K) so
// that only a few are timed -- a model-guided replacement for the black-box
// tile/unroll search of Sec. 4.3.  Forward: y = W3 g(W2 g(W1 x + b1) + b2) + b3
// with g(z) = z * Phi(z).  Backward follows the chain rule; each block
// writes the gradient sums of its rows to the workspace and one pass adds the
// blocks in a fixed order (run-to-run identical), then Adam (Kingma & Ba
// 2015, Algorithm 1) updates the parameters.
//
// Parameter layout (one FP32 buffer, 18817 values): W1 [128][16], b1 [128],
// W2 [128][128], b2 [128], W3 [128], b3 [1].
#include <cuda_runtime.h>

#include "../../include/nk_tune.h"
#include "nk_internal.cuh"

namespace nk {
namespace {

constexpr int D0 = 16, D1 = 128, D2 = 128;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + D1 * D0, OFF_W2 = OFF_B1 + D1, OFF_B2 = OFF_W2 + D2 * D1,
              OFF_W3 = OFF_B2 + D2, OFF_B3 = OFF_W3 + D2, NPARAM = OFF_B3 + 1;
constexpr int ROWS = 8;       // batch rows of one step of a block
constexpr int THREADS = 256;  // hidden unit tid % 128, rows 4 * (tid / 128) .. + 3
constexpr int MAX_BLOCKS = 152;   // blocks of a gradient (one per SM): each loops over its rows

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z) {
  const float Phi = 0.5f * (1.f + erff(z * 0.70710678118654752f));
  const float phi = 0.39894228040143268f * expf(-0.5f * z * z);
  return Phi + z * phi;
}

struct Smem {
  float w2t[D1][D2 + 1];  // W2 transposed, padded: w2t[i][j] = W2[j][i]
  float w1[D1][D0 + 1];
  float x[ROWS][D0];
  float z1[ROWS][D1];
  float z2[ROWS][D2];
  float h1[ROWS][D1];
  float dz2[ROWS][D2];    // dL/dz2
  float dz1[ROWS][D1];    // dL/dz1
  float h1t[D1][ROWS];    // transposed copies: four rows of a unit in one 16-byte load
  float dz2t[D2][ROWS];
  float part[ROWS][4];    // a row's output, summed per warp
  float dy[ROWS];
  float sq[ROWS];
};

__device__ void load_weights(const float* P, Smem& s) {
  const int t = threadIdx.x;
#pragma unroll 8
  for (int e = t; e < D1 * D2; e += THREADS) s.w2t[e % D1][e / D1] = P[OFF_W2 + e];
#pragma unroll
  for (int e = t; e < D1 * D0; e += THREADS) s.w1[e / D0][e % D0] = P[OFF_W1 + e];
}

// Forward for rows r0 .. r0 + 7; fills s.x, z1, h1, h1t, z2.  y[q] of the
// thread's four rows is h2 * W3 of its hidden unit, and the row's output is
// the sum over s.part[row] plus b3.  Ends with the sums in place.
__device__ __forceinline__ void forward_rows(const float* X, int64_t B, int64_t r0, float b1, float b2,
                                             float w3, Smem& s, float (&h2)[4]) {
  const int t = threadIdx.x, j = t & 127, rq = (t >> 7) * 4;
  const float xv = t < ROWS * D0 && r0 + t / D0 < B ? X[r0 * D0 + t] : 0.f;   // under way across the barrier
  __syncthreads();   // the step before has read everything (first step: the weights are in)
  if (t < ROWS * D0) s.x[t / D0][t % D0] = xv;
  __syncthreads();
  float h[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float z = b1;
#pragma unroll
    for (int i = 0; i < D0; ++i) z = fmaf(s.x[rq + q][i], s.w1[j][i], z);
    h[q] = gelu(z);
    s.z1[rq + q][j] = z;
    s.h1[rq + q][j] = h[q];
  }
  *reinterpret_cast<float4*>(&s.h1t[j][rq]) = make_float4(h[0], h[1], h[2], h[3]);
  __syncthreads();
  float z[4] = {b2, b2, b2, b2};
#pragma unroll 16
  for (int i = 0; i < D1; ++i) {
    const float w = s.w2t[i][j];
    const float4 hv = *reinterpret_cast<const float4*>(&s.h1t[i][rq]);
    z[0] = fmaf(hv.x, w, z[0]);
    z[1] = fmaf(hv.y, w, z[1]);
    z[2] = fmaf(hv.z, w, z[2]);
    z[3] = fmaf(hv.w, w, z[3]);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    s.z2[rq + q][j] = z[q];
    h2[q] = gelu(z[q]);
    float a = h2[q] * w3;
#pragma unroll
    for (int o = 16; o; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if ((t & 31) == 0) s.part[rq + q][(t >> 5) & 3] = a;
  }
  __syncthreads();
}

__device__ __forceinline__ float row_output(const Smem& s, int r, float b3) {
  return ((s.part[r][0] + s.part[r][1]) + (s.part[r][2] + s.part[r][3])) + b3;
}

__global__ void __launch_bounds__(THREADS) mlp_forward_kernel(const float* P, const float* X, int64_t B,
                                                              float* __restrict__ y) {
  nk::pdl_wait();      // earlier kernels on the stream have finished
  nk::pdl_trigger();
  extern __shared__ __align__(16) uint8_t raw[];
  Smem& s = *reinterpret_cast<Smem*>(raw);
  const int t = threadIdx.x, j = t & 127;
  load_weights(P, s);
  const float b1 = P[OFF_B1 + j], b2 = P[OFF_B2 + j], w3 = P[OFF_W3 + j], b3 = P[OFF_B3];
  for (int64_t r0 = (int64_t)blockIdx.x * ROWS; r0 < B; r0 += (int64_t)gridDim.x * ROWS) {
    float h2[4];
    forward_rows(X, B, r0, b1, b2, w3, s, h2);
    if (t < ROWS && r0 + t < B) y[r0 + t] = row_output(s, t, b3);
  }
}

// Forward + backward of the MSE loss for the block's rows, eight at a time;
// the block's gradient sums stay in registers (64 values of W2 a thread) and
// go to part[block] once, with its sum of squared errors.
//
// The work is small (114 MFLOP at a batch of 1024: 1.5 us of FP32 FMAs), so
// latency bounds it: 8-row steps give a batch of 1024 128 blocks of eight
// warps, where 32-row blocks gave 32 of four with serial loops over rows and
// units.  A training step (gradient, reduce, Adam) on 1024 rows: 102 -> 21 us.
__global__ void __launch_bounds__(THREADS) mlp_grad_kernel(const float* P, const float* X, const float* T, int64_t B,
                                                           float* __restrict__ part) {
  nk::pdl_wait();      // earlier kernels on the stream have finished
  nk::pdl_trigger();
  extern __shared__ __align__(16) uint8_t raw[];
  Smem& s = *reinterpret_cast<Smem*>(raw);
  const int t = threadIdx.x, j = t & 127, half = t >> 7, rq = half * 4;
  const int jt = (t >> 4) * 8, it = (t & 15) * 4;   // W2 block of this thread: rows jt.., columns it.. and 64 + it..
  load_weights(P, s);
  const float b1 = P[OFF_B1 + j], b2 = P[OFF_B2 + j], w3 = P[OFF_W3 + j], b3 = P[OFF_B3];
  const float inv2b = 2.f / (float)B;
  float gw2[8][8], gw1[D0 / 2];
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int c = 0; c < 8; ++c) gw2[a][c] = 0.f;
#pragma unroll
  for (int k = 0; k < D0 / 2; ++k) gw1[k] = 0.f;
  float gw3 = 0.f, gb2 = 0.f, gb1 = 0.f, gb3 = 0.f, gsq = 0.f;
  for (int64_t r0 = (int64_t)blockIdx.x * ROWS; r0 < B; r0 += (int64_t)gridDim.x * ROWS) {
    float h2[4];
    const bool ok = t < ROWS && r0 + t < B;
    const float target = ok ? T[r0 + t] : 0.f;
    forward_rows(X, B, r0, b1, b2, w3, s, h2);
    if (t < ROWS) {
      const float d = ok ? row_output(s, t, b3) - target : 0.f;
      s.dy[t] = inv2b * d;
      s.sq[t] = d * d;
    }
    __syncthreads();
    float dz[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {   // dL/dz2, gradients of W3 and b2 over this thread's rows
      const float dy = s.dy[rq + q];
      gw3 = fmaf(dy, h2[q], gw3);
      dz[q] = dy * w3 * gelu_grad(s.z2[rq + q][j]);
      gb2 += dz[q];
      s.dz2[rq + q][j] = dz[q];
    }
    *reinterpret_cast<float4*>(&s.dz2t[j][rq]) = make_float4(dz[0], dz[1], dz[2], dz[3]);
    if (t == 0)
      for (int r = 0; r < ROWS; ++r) { gb3 += s.dy[r]; gsq += s.sq[r]; }
    __syncthreads();
    // gW2[jj][i] += dz2[r][jj] h1[r][i]
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      const float4 d0 = *reinterpret_cast<const float4*>(&s.dz2[r][jt]);
      const float4 d1 = *reinterpret_cast<const float4*>(&s.dz2[r][jt + 4]);
      const float4 v0 = *reinterpret_cast<const float4*>(&s.h1[r][it]);
      const float4 v1 = *reinterpret_cast<const float4*>(&s.h1[r][64 + it]);
      const float dd[8] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
      const float hh[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
#pragma unroll
      for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int c = 0; c < 8; ++c) gw2[a][c] = fmaf(dd[a], hh[c], gw2[a][c]);
    }
    // dL/dh1[r][i] = sum_jj dz2[r][jj] W2[jj][i], then dL/dz1, for i = j
    float dh[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 16
    for (int jj = 0; jj < D2; ++jj) {
      const float w = s.w2t[j][jj];
      const float4 dv = *reinterpret_cast<const float4*>(&s.dz2t[jj][rq]);
      dh[0] = fmaf(dv.x, w, dh[0]);
      dh[1] = fmaf(dv.y, w, dh[1]);
      dh[2] = fmaf(dv.z, w, dh[2]);
      dh[3] = fmaf(dv.w, w, dh[3]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float d = dh[q] * gelu_grad(s.z1[rq + q][j]);
      gb1 += d;
      s.dz1[rq + q][j] = d;
    }
    __syncthreads();
    // gW1[j][k] += dz1[r][j] x[r][k]: this thread's half of the inputs
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      const float d = s.dz1[r][j];
#pragma unroll
      for (int k = 0; k < D0 / 2; ++k) gw1[k] = fmaf(d, s.x[r][half * (D0 / 2) + k], gw1[k]);
    }
  }
  // the two halves of the block hold different rows of gW3, gb2 and gb1
  __syncthreads();
  if (half) {
    s.z1[0][j] = gw3;
    s.z1[1][j] = gb2;
    s.z1[2][j] = gb1;
  }
  __syncthreads();
  float* g = part + (int64_t)blockIdx.x * (NPARAM + 1);
  if (!half) {
    g[OFF_W3 + j] = gw3 + s.z1[0][j];
    g[OFF_B2 + j] = gb2 + s.z1[1][j];
    g[OFF_B1 + j] = gb1 + s.z1[2][j];
  }
  if (t == 0) {
    g[OFF_B3] = gb3;
    g[NPARAM] = gsq;
  }
#pragma unroll
  for (int k = 0; k < D0 / 2; ++k) g[OFF_W1 + j * D0 + half * (D0 / 2) + k] = gw1[k];
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int c = 0; c < 8; ++c) g[OFF_W2 + (jt + a) * D1 + (c / 4) * 64 + it + (c % 4)] = gw2[a][c];
}

// grad[p] = sum_b part[b][p]; loss = sum_b part[b][NPARAM] / B.  Four threads
// a parameter sum every fourth block in order and are added in a fixed tree,
// so the result is the same every run; sixteen loads in flight a thread.
constexpr int RED_P = 64;
__global__ void __launch_bounds__(4 * RED_P) mlp_reduce_kernel(const float* part, int nblocks, int64_t B,
                                                               float* __restrict__ grad, float* __restrict__ loss) {
  nk::pdl_wait();      // earlier kernels on the stream have finished
  nk::pdl_trigger();
  __shared__ float sm[4][RED_P];
  const int lp = threadIdx.x % RED_P, q = threadIdx.x / RED_P;
  const int p = blockIdx.x * RED_P + lp;
  float a = 0.f;
  if (p <= NPARAM) {
#pragma unroll 16
    for (int b = q; b < nblocks; b += 4) a += part[(int64_t)b * (NPARAM + 1) + p];
  }
  sm[q][lp] = a;
  __syncthreads();
  if (q || p > NPARAM) return;
  a = (sm[0][lp] + sm[1][lp]) + (sm[2][lp] + sm[3][lp]);
  if (p < NPARAM) grad[p] = a;
  else if (loss) *loss = a / (float)B;
}

__global__ void mlp_adam_kernel(float* __restrict__ P, const float* g, float* __restrict__ m,
                                float* __restrict__ v, int n, float lr, float b1, float b2, float eps,
                                float bc1, float bc2) {
  nk::pdl_wait();      // earlier kernels on the stream have finished
  nk::pdl_trigger();
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const float gp = g[p];
  const float mp = b1 * m[p] + (1.f - b1) * gp;
  const float vp = b2 * v[p] + (1.f - b2) * gp * gp;
  m[p] = mp;
  v[p] = vp;
  const float mh = mp / bc1;
  const float vh = vp / bc2;
  P[p] -= lr * mh / (sqrtf(vh) + eps);
}

// Blocks of a batch: eight rows each until every SM has one.
int64_t blocks_of(int64_t B) {
  const int64_t nb = (B + ROWS - 1) / ROWS;
  return nb < MAX_BLOCKS ? nb : MAX_BLOCKS;
}

nk_status set_smem(const void* fn) {
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
  return e == cudaSuccess ? NK_OK : cuda_fail(e, "cudaFuncSetAttribute(mlp)");
}

}  // namespace
}  // namespace nk

using namespace nk;

extern "C" {

size_t nk_mlp_param_count(void) { return NPARAM; }

size_t nk_mlp_workspace_size(int64_t B) {
  return (size_t)blocks_of(B) * (NPARAM + 1) * sizeof(float);
}

nk_status nk_mlp_forward(const float* params, const float* X, int64_t B, float* y, void* stream) {
  nk::NvtxRange nvtx_range_("nk_mlp_forward");
  nk_status s = require_device();
  if (s != NK_OK) return s;
  if (B < 0) return fail(NK_ERR_INVALID_ARG, "negative batch");
  if (B == 0) return NK_OK;
  if (!params || !X || !y) return fail(NK_ERR_INVALID_ARG, "null pointer");
  if ((s = set_smem(reinterpret_cast<const void*>(mlp_forward_kernel))) != NK_OK) return s;
  const int64_t nb = blocks_of(B);
  (void)nk::launch_k(mlp_forward_kernel, dim3((unsigned)nb), dim3(THREADS), sizeof(Smem), static_cast<cudaStream_t>(stream), 1, params, X, B, y);
  return check_launch("mlp_forward_kernel");
}

nk_status nk_mlp_grad(const float* params, const float* X, const float* t, int64_t B, float* grad, float* loss,
                      void* ws, size_t ws_bytes, void* stream) {
  nk::NvtxRange nvtx_range_("nk_mlp_grad");
  nk_status s = require_device();
  if (s != NK_OK) return s;
  if (B <= 0) return fail(NK_ERR_INVALID_ARG, "batch must be positive");
  if (!params || !X || !t || !grad) return fail(NK_ERR_INVALID_ARG, "null pointer");
  if (!ws || ws_bytes < nk_mlp_workspace_size(B))
    return fail(NK_ERR_WORKSPACE, "mlp gradient needs %zu bytes of workspace", nk_mlp_workspace_size(B));
  if ((s = set_smem(reinterpret_cast<const void*>(mlp_grad_kernel))) != NK_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int64_t nb = blocks_of(B);
  float* part = static_cast<float*>(ws);
  (void)nk::launch_k(mlp_grad_kernel, dim3((unsigned)nb), dim3(THREADS), sizeof(Smem), st, 1, params, X, t, B, part);
  if ((s = check_launch("mlp_grad_kernel")) != NK_OK) return s;
  (void)nk::launch_k(mlp_reduce_kernel, dim3((NPARAM + 1 + RED_P - 1) / RED_P), dim3(4 * RED_P), 0, st, 1, part, (int)nb, B, grad,
                     loss);
  return check_launch("mlp_reduce_kernel");
}

nk_status nk_mlp_adam(float* params, const float* grad, float* m, float* v, int32_t step, float lr, float beta1,
                      float beta2, float eps, void* stream) {
  nk::NvtxRange nvtx_range_("nk_mlp_adam");
  nk_status s = require_device();
  if (s != NK_OK) return s;
  if (step < 1) return fail(NK_ERR_INVALID_ARG, "Adam step counts from 1");
  if (!params || !grad || !m || !v) return fail(NK_ERR_INVALID_ARG, "null pointer");
  const float bc1 = 1.f - powf(beta1, (float)step);
  const float bc2 = 1.f - powf(beta2, (float)step);
  (void)nk::launch_k(mlp_adam_kernel, dim3((NPARAM + 255) / 256), dim3(256), 0, static_cast<cudaStream_t>(stream), 1, 
      params, grad, m, v, NPARAM, lr, beta1, beta2, eps, bc1, bc2);
  return check_launch("mlp_adam_kernel");
}

}  // extern "C"
