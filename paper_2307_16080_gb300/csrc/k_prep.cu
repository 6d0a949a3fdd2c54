// k_prep.cu -- operand preparation and the validation norm.
//
// Operand prep turns FP32 operands into what the tensor cores read:
//   BF16     x -> bf16_rn(x)
//   FP8      s = 448/amax(|x|) (1 if amax is 0 or not finite), q = e4m3_rn_sat(x*s)
//   BF16x3   hi = bf16_rn(x), lo = bf16_rn(x - hi)
// optionally transposing [rows, cols] -> [cols, rows] so that a [K,N] operand
// becomes K-major.  These passes are HBM-bound: 128-bit loads, one read and
// one write of every element, 64x64 shared-memory tiles for the transpose.
// Rounding uses CUDA's own conversion intrinsics (RNE; satfinite for E4M3).
//
// The validation norm sums (C-R)^2 and R^2 in FP64 over a fixed partition
// (fixed block count, fixed tree), so its result is identical run to run.
#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>

#include "nk_internal.cuh"

namespace nk {
namespace {

constexpr int kAmaxBlocks = 1024;
constexpr int kNormBlocks = 1024;

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Prologue program on four consecutive elements starting at offset `off`.
template <bool PRO>
__device__ __forceinline__ void pro4(const EwProg& e, float* v, int64_t off) {
  if constexpr (PRO) {
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = ew_run(e, v[j], off + j);
  }
}

// amax over a [rows, cols] matrix with row stride ld.  Stage 1: one partial
// per block; stage 2: one block folds the partials.  NaN inputs make the
// result NaN (the scale then falls back to 1).  PRO: the amax of the values
// after the prologue program `pro`.
// Registers for five blocks an SM: four (52 registers) take 43.9 us instead of
// 39.8 for 268 MB.
template <bool PRO>
__global__ void __launch_bounds__(256, PRO ? 2 : 5) amax_stage1(const float* x, int64_t rows, int64_t cols, int64_t ld,
                                                                float* __restrict__ partial,
                                                                const __grid_constant__ EwProg pro) {
  nk::pdl_wait();      // earlier kernels on the stream have finished
  nk::pdl_trigger();
  float m = 0.f;
  bool nan = false;
  const bool al = (reinterpret_cast<uintptr_t>(x) & 15) == 0;
  if (al && ld == cols && (rows * cols) % 4 == 0) {
    // dense: one flat run of float4, no index arithmetic per element
    const float4* x4 = reinterpret_cast<const float4*>(x);
    const int64_t n4 = rows * cols / 4;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    auto fold = [&](float4 v, int64_t i) {
      if constexpr (PRO) {
        float w[4] = {v.x, v.y, v.z, v.w};
        pro4<PRO>(pro, w, 4 * i);
        v = make_float4(w[0], w[1], w[2], w[3]);
      }
      nan |= (v.x != v.x) | (v.y != v.y) | (v.z != v.z) | (v.w != v.w);
      m = fmaxf(m, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
    };
    // eight loads in flight a thread (67 MB: 12.6 us; 13.2 with one)
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (; i + 7 * stride < n4; i += 8 * stride) {
      float4 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = x4[i + u * stride];
#pragma unroll
      for (int u = 0; u < 8; ++u) fold(v[u], i + u * stride);
    }
    // and in the last, partial round (3 M values: 3.8 us, 4.8 one by one)
    float4 v[7];
#pragma unroll
    for (int u = 0; u < 7; ++u)
      if (i + u * stride < n4) v[u] = x4[i + u * stride];
#pragma unroll
    for (int u = 0; u < 7; ++u)
      if (i + u * stride < n4) fold(v[u], i + u * stride);
  } else {
    // strided rows: blocks stride over rows, threads over the row
    const bool vec = al && (cols % 4 == 0) && (ld % 4 == 0);
    for (int64_t r = blockIdx.x; r < rows; r += gridDim.x) {
      const float* row = x + r * ld;
      if (vec) {
        for (int64_t c = threadIdx.x; c < cols / 4; c += blockDim.x) {
          float4 v = reinterpret_cast<const float4*>(row)[c];
          if constexpr (PRO) {
            float w[4] = {v.x, v.y, v.z, v.w};
            pro4<PRO>(pro, w, r * ld + 4 * c);
            v = make_float4(w[0], w[1], w[2], w[3]);
          }
          nan |= (v.x != v.x) | (v.y != v.y) | (v.z != v.z) | (v.w != v.w);
          m = fmaxf(m, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
        }
      } else {
        for (int64_t c = threadIdx.x; c < cols; c += blockDim.x) {
          float v = row[c];
          if constexpr (PRO) v = ew_run(pro, v, r * ld + c);
          nan |= (v != v);
          m = fmaxf(m, fabsf(v));
        }
      }
    }
  }
  if (__any_sync(0xffffffffu, nan)) m = __int_as_float(0x7fc00000);
  __shared__ float sm[32];
  float w = warp_max(m);
  bool wn = __any_sync(0xffffffffu, m != m);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x / 32] = wn ? __int_as_float(0x7fc00000) : w;
  __syncthreads();
  if (threadIdx.x < 32) {
    const int nw = blockDim.x / 32;
    float v = threadIdx.x < nw ? sm[threadIdx.x] : 0.f;
    bool bn = __any_sync(0xffffffffu, v != v);
    v = warp_max(v);
    if (threadIdx.x == 0) partial[blockIdx.x] = bn ? __int_as_float(0x7fc00000) : v;
  }
}

__global__ void amax_stage2(const float* partial, int n, float* __restrict__ out) {
  nk::pdl_wait();      // earlier kernels on the stream have finished
  nk::pdl_trigger();
  float m = 0.f;
  bool nan = false;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    float v = partial[i];
    nan |= (v != v);
    m = fmaxf(m, v);
  }
  __shared__ float sm[32];
  __shared__ int sn;
  if (threadIdx.x == 0) sn = 0;
  __syncthreads();
  if (nan) atomicOr(&sn, 1);
  float w = warp_max(m);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x / 32] = w;
  __syncthreads();
  if (threadIdx.x < 32) {
    float v = threadIdx.x < (int)(blockDim.x / 32) ? sm[threadIdx.x] : 0.f;
    v = warp_max(v);
    if (threadIdx.x == 0) *out = sn ? __int_as_float(0x7fc00000) : v;
  }
}

__device__ __forceinline__ float fp8_scale_of(const float* amax) {
  const float a = *amax;
  return (a > 0.f && a <= 3.402823466e38f) ? __fdiv_rn(448.f, a) : 1.f;
}

// One element of each cast kind.  kind 0: bf16, 1: e4m3, 2: bf16 hi/lo.
template <int KIND>
struct Caster;

template <>
struct Caster<0> {
  using T = __nv_bfloat16;
  __device__ static void cvt(float x, float, T& o0, T&) { o0 = __float2bfloat16_rn(x); }
};
template <>
struct Caster<1> {
  using T = __nv_fp8_storage_t;
  __device__ static void cvt(float x, float s, T& o0, T&) {
    o0 = __nv_cvt_float_to_fp8(__fmul_rn(x, s), __NV_SATFINITE, __NV_E4M3);
  }
};
template <>
struct Caster<2> {
  using T = __nv_bfloat16;
  __device__ static void cvt(float x, float, T& o0, T& o1) {
    o0 = __float2bfloat16_rn(x);
    o1 = __float2bfloat16_rn(__fsub_rn(x, __bfloat162float(o0)));
  }
};

// Row-major cast whose output rows take no word stores: neighbouring lanes take
// neighbouring elements, eight each, 2^tx_log apart.
template <int KIND, bool PRO>
__global__ void __launch_bounds__(256) cast_rows_single(const float* in, int64_t rows, int64_t cols, int64_t ld_in,
                                                        const float* amax, typename Caster<KIND>::T* __restrict__ o0,
                                                        typename Caster<KIND>::T* __restrict__ o1, int64_t ld_out,
                                                        float* scale_out, int tx_log, const __grid_constant__ EwProg pro) {
  nk::pdl_wait();      // earlier kernels on the stream have finished
  nk::pdl_trigger();
  using T = typename Caster<KIND>::T;
  constexpr int V = 8;
  const float s = KIND == 1 ? fp8_scale_of(amax) : 1.f;
  if (scale_out && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *scale_out = s;
  const int ty = 256 >> tx_log;
  const int64_t c = ((int64_t)blockIdx.x << tx_log) * V + (threadIdx.x & ((1 << tx_log) - 1));
  for (int64_t r = (int64_t)blockIdx.y * ty + (threadIdx.x >> tx_log); r < rows; r += (int64_t)gridDim.y * ty) {
    float v[V];
#pragma unroll
    for (int j = 0; j < V; ++j) v[j] = c + (j << tx_log) < cols ? in[r * ld_in + c + (j << tx_log)] : 0.f;
#pragma unroll
    for (int j = 0; j < V; ++j) {
      const int64_t cc = c + (j << tx_log);
      if (cc >= cols) break;
      if constexpr (PRO) v[j] = ew_run(pro, v[j], r * ld_in + cc);
      T a, b;
      Caster<KIND>::cvt(v[j], s, a, b);
      o0[r * ld_out + cc] = a;
      if (KIND == 2) o1[r * ld_out + cc] = b;
    }
  }
}

// Row-major cast without transpose: eight elements per thread per step, read
// as two 16-byte words (one by one where the input's alignment does not allow
// it) and written as one 16-byte word of BF16 (8 bytes of E4M3).  HBM-bound; a
// block is 2^tx_log chunks of a row by as many rows as fit, so no index needs
// a division and short rows fill a block.  Per-element 2-byte stores and a
// 64-bit division per four elements took 21.2 us for the hi / lo split of 3001
// x 1999 (48 MB), now 10.5; BF16 of 8192^2 (402 MB) 64 us, now 54.
// PRO: the prologue program `pro` runs on each element before the cast.
template <int KIND, bool PRO>
__global__ void __launch_bounds__(256) cast_rows(const float* in, int64_t rows, int64_t cols, int64_t ld_in,
                                                 const float* amax, typename Caster<KIND>::T* __restrict__ o0,
                                                 typename Caster<KIND>::T* __restrict__ o1, int64_t ld_out,
                                                 float* scale_out, int tx_log, const __grid_constant__ EwProg pro) {
  nk::pdl_wait();      // earlier kernels on the stream have finished
  nk::pdl_trigger();
  using T = typename Caster<KIND>::T;
  constexpr int V = 8;
  const float s = KIND == 1 ? fp8_scale_of(amax) : 1.f;
  if (scale_out && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *scale_out = s;
  constexpr int OB = V * (int)sizeof(T);   // bytes of an output word: 16 (BF16) or 8 (E4M3)
  const int64_t c = (((int64_t)blockIdx.x << tx_log) + (threadIdx.x & ((1 << tx_log) - 1))) * V;
  const int ty = 256 >> tx_log;
  if (c >= cols) return;
  const bool whole = c + V <= cols;
  const bool vin = whole && (ld_in % 4 == 0) && ((reinterpret_cast<uintptr_t>(in) & 15) == 0);
  for (int64_t r = (int64_t)blockIdx.y * ty + (threadIdx.x >> tx_log); r < rows; r += (int64_t)gridDim.y * ty) {
    const float* src = in + r * ld_in + c;
    float v[V];
    if (vin) {
      const float4 q0 = *reinterpret_cast<const float4*>(src), q1 = *reinterpret_cast<const float4*>(src + 4);
      v[0] = q0.x; v[1] = q0.y; v[2] = q0.z; v[3] = q0.w;
      v[4] = q1.x; v[5] = q1.y; v[6] = q1.z; v[7] = q1.w;
    } else {
#pragma unroll
      for (int j = 0; j < V; ++j) v[j] = c + j < cols ? src[j] : 0.f;
    }
    if constexpr (PRO) {
#pragma unroll
      for (int j = 0; j < V; ++j)
        if (c + j < cols) v[j] = ew_run(pro, v[j], r * ld_in + c + j);
    }
    __align__(16) T a[V];
    __align__(16) T b[V];
#pragma unroll
    for (int j = 0; j < V; ++j) Caster<KIND>::cvt(v[j], s, a[j], b[j]);
    T* d0 = o0 + r * ld_out + c;
    if (whole) {
      if constexpr (OB == 16) {
        *reinterpret_cast<uint4*>(d0) = *reinterpret_cast<const uint4*>(a);
        if (KIND == 2) *reinterpret_cast<uint4*>(o1 + r * ld_out + c) = *reinterpret_cast<const uint4*>(b);
      } else {
        *reinterpret_cast<uint2*>(d0) = *reinterpret_cast<const uint2*>(a);
      }
    } else {
#pragma unroll
      for (int j = 0; j < V; ++j) {
        if (c + j < cols) {
          d0[j] = a[j];
          if (KIND == 2) o1[r * ld_out + c + j] = b[j];
        }
      }
    }
  }
}

// Transposing cast of a matrix with few rows or few columns, most of whose
// tile below would be empty: a thread takes one position of the long side and
// walks the short one.  us, with the tile / this: 3 x 1000000 to E4M3 57 / 9,
// 1000000 x 3 33 / 13.
template <int KIND, bool PRO>
__global__ void __launch_bounds__(256) cast_transpose_few(const float* in, int64_t rows, int64_t cols, int64_t ld_in,
                                                          const float* amax,
                                                          typename Caster<KIND>::T* __restrict__ o0,
                                                          typename Caster<KIND>::T* __restrict__ o1, int64_t ld_out,
                                                          float* scale_out, bool few_rows,
                                                          const __grid_constant__ EwProg pro) {
  nk::pdl_wait();      // earlier kernels on the stream have finished
  nk::pdl_trigger();
  using T = typename Caster<KIND>::T;
  const float s = KIND == 1 ? fp8_scale_of(amax) : 1.f;
  if (scale_out && blockIdx.x == 0 && threadIdx.x == 0) *scale_out = s;
  const int64_t n = few_rows ? cols : rows;
  const int m = (int)(few_rows ? rows : cols);
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256)
#pragma unroll 4
    for (int k = 0; k < m; ++k) {
      const int64_t r = few_rows ? k : i, c = few_rows ? i : k;
      float v = in[r * ld_in + c];
      if constexpr (PRO) v = ew_run(pro, v, r * ld_in + c);
      T a, b;
      Caster<KIND>::cvt(v, s, a, b);
      o0[c * ld_out + r] = a;
      if (KIND == 2) o1[c * ld_out + r] = b;
    }
}

// Transposing cast: a tile of 64 input columns by 32 words of P rows through
// shared memory, where a word holds the P converted values of one column (2
// BF16 or 4 E4M3: P input rows).  Converting first means a thread stores four
// columns' words at once and gathers 16 output bytes from four words.  Reads
// are 128-bit along the input rows, writes 16 bytes a lane and 128 contiguous
// bytes per output row; quads of columns are xor-swizzled by the word row, so
// neither side has a bank conflict.  HBM-bound: 8192^2 to BF16 (402 MB) 70 us
// with an FP32 tile and two-way conflicts, now 53.
template <int KIND, bool PRO>
__global__ void __launch_bounds__(256) cast_transpose(const float* in, int64_t rows, int64_t cols,
                                                      int64_t ld_in, const float* amax,
                                                      typename Caster<KIND>::T* __restrict__ o0,
                                                      typename Caster<KIND>::T* __restrict__ o1, int64_t ld_out,
                                                      float* scale_out, const __grid_constant__ EwProg pro) {
  nk::pdl_wait();      // earlier kernels on the stream have finished
  nk::pdl_trigger();
  using T = typename Caster<KIND>::T;
  constexpr int P = 4 / (int)sizeof(T);             // values (input rows) of a word
  constexpr int TR = 32 * P, TC = 64, VEC = 4 * P;  // VEC: output elements of a 16-byte store
  constexpr int OUTS = KIND == 2 ? 2 : 1;
  __shared__ __align__(16) uint32_t tile[OUTS][32][TC];
  const float s = KIND == 1 ? fp8_scale_of(amax) : 1.f;
  if (scale_out && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *scale_out = s;
  const int t = threadIdx.x;
  const int64_t r0 = (int64_t)blockIdx.y * TR, c0 = (int64_t)blockIdx.x * TC;
  const bool vin = (ld_in % 4 == 0) && ((reinterpret_cast<uintptr_t>(in) & 15) == 0) && c0 + TC <= cols;
  const int cc = (t % 16) * 4;
  float v[2][P][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int h = 0; h < P; ++h) {
      const int64_t r = r0 + (t / 16 + 16 * i) * P + h, c = c0 + cc;
      float* x = v[i][h];
      x[0] = x[1] = x[2] = x[3] = 0.f;
      if (r < rows) {
        if (vin) {
          const float4 q = *reinterpret_cast<const float4*>(in + r * ld_in + c);
          x[0] = q.x; x[1] = q.y; x[2] = q.z; x[3] = q.w;
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (c + j < cols) x[j] = in[r * ld_in + c + j];
        }
      }
    }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int g = t / 16 + 16 * i;
    __align__(16) T w0[4][P];
    __align__(16) T w1[4][P];
#pragma unroll
    for (int h = 0; h < P; ++h)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if constexpr (PRO) {
          const int64_t r = r0 + g * P + h, c = c0 + cc + j;
          if (r < rows && c < cols) v[i][h][j] = ew_run(pro, v[i][h][j], r * ld_in + c);
        }
        Caster<KIND>::cvt(v[i][h][j], s, w0[j][h], w1[j][h]);
      }
    const int at = ((t % 16) ^ (g >> 2)) * 4;
    *reinterpret_cast<uint4*>(&tile[0][g][at]) = *reinterpret_cast<const uint4*>(w0);
    if constexpr (KIND == 2) *reinterpret_cast<uint4*>(&tile[1][g][at]) = *reinterpret_cast<const uint4*>(w1);
  }
  __syncthreads();
  // output row c0 + oc holds input column oc; its elements are input rows r0 ..
  const bool vout = ((ld_out * (int64_t)sizeof(T)) % 16 == 0) &&
                    ((reinterpret_cast<uintptr_t>(o0) & 15) == 0) &&
                    (KIND != 2 || (reinterpret_cast<uintptr_t>(o1) & 15) == 0);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int idx = t + 256 * i;
    const int chunk = idx % 8, oc = idx / 8;
    const int64_t orow = c0 + oc, ocol = r0 + chunk * VEC;
    if (orow >= cols) continue;
#pragma unroll
    for (int q = 0; q < OUTS; ++q) {
      uint4 w;
      const int at = ((oc >> 2) ^ chunk) * 4 + (oc & 3);
      w.x = tile[q][chunk * 4 + 0][at];
      w.y = tile[q][chunk * 4 + 1][at];
      w.z = tile[q][chunk * 4 + 2][at];
      w.w = tile[q][chunk * 4 + 3][at];
      T* d = (q ? o1 : o0) + orow * ld_out + ocol;
      if (vout && ocol + VEC <= rows) {
        *reinterpret_cast<uint4*>(d) = w;
      } else {
        __align__(16) T a[VEC];
        *reinterpret_cast<uint4*>(a) = w;
#pragma unroll
        for (int j = 0; j < VEC; ++j)
          if (ocol + j < rows) d[j] = a[j];
      }
    }
  }
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Fixed-order FP64 block sums: thread i of block b visits elements
// b*blockDim + i + k*gridDim*blockDim; warp tree, then a tree over warps.
__global__ void norm_stage1(const float* C, int64_t ldc, const double* R,
                            int64_t ldr, int64_t M, int64_t N, double* __restrict__ partial) {
  nk::pdl_wait();      // earlier kernels on the stream have finished
  nk::pdl_trigger();
  double e = 0.0, r2 = 0.0;
  const int64_t total = M * N;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t m = i / N, n = i % N;
    const double r = R[m * ldr + n];
    const double d = (double)C[m * ldc + n] - r;
    e = fma(d, d, e);
    r2 = fma(r, r, r2);
  }
  __shared__ double se[32], sr[32];
  e = warp_sum_d(e);
  r2 = warp_sum_d(r2);
  if ((threadIdx.x & 31) == 0) { se[threadIdx.x / 32] = e; sr[threadIdx.x / 32] = r2; }
  __syncthreads();
  if (threadIdx.x < 32) {
    const int nw = blockDim.x / 32;
    double a = threadIdx.x < nw ? se[threadIdx.x] : 0.0;
    double b = threadIdx.x < nw ? sr[threadIdx.x] : 0.0;
    a = warp_sum_d(a);
    b = warp_sum_d(b);
    if (threadIdx.x == 0) { partial[2 * blockIdx.x] = a; partial[2 * blockIdx.x + 1] = b; }
  }
}

__global__ void norm_stage2(const double* partial, int n, double* __restrict__ out) {
  nk::pdl_wait();      // earlier kernels on the stream have finished
  nk::pdl_trigger();
  double e = 0.0, r2 = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) { e += partial[2 * i]; r2 += partial[2 * i + 1]; }
  __shared__ double se[32], sr[32];
  e = warp_sum_d(e);
  r2 = warp_sum_d(r2);
  if ((threadIdx.x & 31) == 0) { se[threadIdx.x / 32] = e; sr[threadIdx.x / 32] = r2; }
  __syncthreads();
  if (threadIdx.x < 32) {
    const int nw = blockDim.x / 32;
    double a = threadIdx.x < nw ? se[threadIdx.x] : 0.0;
    double b = threadIdx.x < nw ? sr[threadIdx.x] : 0.0;
    a = warp_sum_d(a);
    b = warp_sum_d(b);
    if (threadIdx.x == 0) { out[0] = a; out[1] = b; }
  }
}

template <int KIND, bool PRO>
nk_status launch_cast(const float* in, int64_t rows, int64_t cols, int64_t ld_in,
                      const float* amax, void* out0, void* out1, int64_t ld_out, int transpose,
                      float* scale_out, cudaStream_t st, int sms, const EwProg& pro) {
  using T = typename Caster<KIND>::T;
  T* o0 = static_cast<T*>(out0);
  T* o1 = static_cast<T*>(out1);
  if (transpose) {
    constexpr int TR = 32 * (4 / (int)sizeof(T));   // rows of a tile (cast_transpose)
    dim3 grid((unsigned)((cols + 63) / 64), (unsigned)((rows + TR - 1) / TR));
    if (grid.y > 65535) return fail(NK_ERR_UNSUPPORTED, "too many rows for the transposing cast");
    const bool few_rows = rows * 4 <= TR && rows <= cols;   // a quarter of a tile
    if (few_rows || cols <= 16) {
      const int64_t blocks = ((few_rows ? cols : rows) + 255) / 256;
      (void)nk::launch_k(cast_transpose_few<KIND, PRO>, dim3((unsigned)std::min<int64_t>(blocks, (int64_t)sms * 64)), dim3(256),
                         0, st, 1, in, rows, cols, ld_in, amax, o0, o1, ld_out, scale_out, few_rows, pro);
      return check_launch("cast kernel");
    }
    (void)nk::launch_k(cast_transpose<KIND, PRO>, dim3(grid), dim3(256), 0, st, 1, in, rows, cols, ld_in, amax, o0, o1, ld_out, scale_out, pro);
  } else {
    // a dense matrix whose rows do not end on words is one long row of them
    // (us: 1001 x 1003 to BF16 3.6 / 1.9, 1000000 x 3 6.4 / 4.4)
    if (ld_in == cols && ld_out == cols && cols % 8 != 0) {
      cols *= rows;
      ld_in = ld_out = cols + (8 - cols % 8) % 8;   // one row: only the alignment of the strides is looked at
      rows = 1;
    }
    const int64_t chunks = (cols + 7) / 8;
    int tx_log = 0;
    while (tx_log < 8 && (int64_t(1) << tx_log) < chunks) ++tx_log;
    const int64_t bx = (chunks + (int64_t(1) << tx_log) - 1) >> tx_log;
    if (bx > INT32_MAX) return fail(NK_ERR_UNSUPPORTED, "too many columns for the cast");
    const int ty = 256 >> tx_log;
    int64_t by = (rows + ty - 1) / ty;
    const int64_t cap = ((int64_t)sms * 32 + bx - 1) / bx;   // a few waves of eight resident blocks
    if (by > cap) by = cap;
    if (by > 65535) by = 65535;
    constexpr uintptr_t OB = 8 * sizeof(T);   // an output word: eight values
    const bool words = ld_out * sizeof(T) % OB == 0 && reinterpret_cast<uintptr_t>(o0) % OB == 0 &&
                       (KIND != 2 || reinterpret_cast<uintptr_t>(o1) % OB == 0);
    (void)nk::launch_k(words ? cast_rows<KIND, PRO> : cast_rows_single<KIND, PRO>, dim3((unsigned)bx, (unsigned)by),
                       dim3(256), 0, st, 1, in, rows, cols, ld_in, amax, o0, o1, ld_out, scale_out, tx_log, pro);
  }
  return check_launch("cast kernel");
}

template <int KIND>
nk_status launch_cast(const float* in, int64_t rows, int64_t cols, int64_t ld_in, const float* amax,
                      void* out0, void* out1, int64_t ld_out, int transpose, float* scale_out, cudaStream_t st,
                      int sms, const EwProg* pro) {
  if (pro && pro->n)
    return launch_cast<KIND, true>(in, rows, cols, ld_in, amax, out0, out1, ld_out, transpose, scale_out, st, sms,
                                   *pro);
  return launch_cast<KIND, false>(in, rows, cols, ld_in, amax, out0, out1, ld_out, transpose, scale_out, st, sms,
                                  EwProg{});
}

// Y = prog(X) over a rank-4 (padded) strided tensor: one element per thread
// per step, grid-stride.  `dense`: X, Y and the operands are one contiguous
// run, handled as float4 (the element offset is the flat index).
__global__ void ew_dense_kernel(const float* x, float* y, int64_t n,
                                const __grid_constant__ EwProg prog) {
  nk::pdl_wait();      // earlier kernels on the stream have finished
  nk::pdl_trigger();
  const int64_t n4 = n / 4;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
    const float4 v = reinterpret_cast<const float4*>(x)[i];
    float4 o;
    o.x = ew_run(prog, v.x, 4 * i);
    o.y = ew_run(prog, v.y, 4 * i + 1);
    o.z = ew_run(prog, v.z, 4 * i + 2);
    o.w = ew_run(prog, v.w, 4 * i + 3);
    reinterpret_cast<float4*>(y)[i] = o;
  }
  for (int64_t i = 4 * n4 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
    y[i] = ew_run(prog, x[i], i);
}

struct Strided4 {
  int64_t shape[4];
  int64_t sx[4], sy[4];
};

__global__ void ew_strided_kernel(const float* x, float* y, int64_t n, const __grid_constant__ Strided4 g,
                                  const __grid_constant__ EwProg prog) {
  nk::pdl_wait();      // earlier kernels on the stream have finished
  nk::pdl_trigger();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    int64_t r = i, ox = 0, oy = 0;
#pragma unroll
    for (int d = 3; d >= 0; --d) {
      const int64_t id = r % g.shape[d];
      r /= g.shape[d];
      ox += id * g.sx[d];
      oy += id * g.sy[d];
    }
    y[oy] = ew_run(prog, x[ox], oy);
  }
}

}  // namespace

size_t prep_amax_ws(int64_t) { return kAmaxBlocks * sizeof(float); }

nk_status prep_amax(const float* x, int64_t rows, int64_t cols, int64_t ld, float* amax, void* ws,
                    size_t ws_bytes, cudaStream_t st, const EwProg* pro) {
  if (!amax) return fail(NK_ERR_INVALID_ARG, "amax: null pointer");
  if (rows * cols == 0) {   // max over nothing: 0 (the scale then falls back to 1)
    cudaError_t e = cudaMemsetAsync(amax, 0, sizeof(float), st);
    return e == cudaSuccess ? NK_OK : cuda_fail(e, "cudaMemsetAsync(amax)");
  }
  if (!x) return fail(NK_ERR_INVALID_ARG, "amax: null pointer");
  if (!ws || ws_bytes < prep_amax_ws(rows * cols))
    return fail(NK_ERR_WORKSPACE, "amax needs %zu bytes of workspace", prep_amax_ws(rows * cols));
  // long runs fill whole rounds of eight words; shorter ones take one wave of the
  // five blocks an SM holds, and at most four words a thread where these are
  // too many (500 thousand values: 2.8 us, 3.4 with 1024 blocks)
  int sms = 0;
  nk_status s = require_device(&sms);
  if (s != NK_OK) return s;
  int blocks = rows * cols >= int64_t(kAmaxBlocks) * 256 * 32 ? kAmaxBlocks : std::min(kAmaxBlocks, 5 * sms);
  if (ld == cols) blocks = (int)std::min<int64_t>(blocks, (rows * cols + 4095) / 4096);
  if (pro && pro->n)
    (void)nk::launch_k(amax_stage1<true>, dim3(blocks), dim3(256), 0, st, 1, x, rows, cols, ld, static_cast<float*>(ws), *pro);
  else
    (void)nk::launch_k(amax_stage1<false>, dim3(blocks), dim3(256), 0, st, 1, x, rows, cols, ld, static_cast<float*>(ws), EwProg{});
  if ((s = check_launch("amax_stage1")) != NK_OK) return s;
  (void)nk::launch_k(amax_stage2, dim3(1), dim3(1024), 0, st, 1, static_cast<float*>(ws), blocks, amax);
  return check_launch("amax_stage2");
}

nk_status prep_cast(int kind, const float* in, int64_t rows, int64_t cols, int64_t ld_in,
                    const float* amax, void* out0, void* out1, int64_t ld_out, int transpose,
                    float* scale_out, cudaStream_t st, const EwProg* pro) {
  int sms = 0;
  nk_status s = require_device(&sms);
  if (s != NK_OK) return s;
  if (rows <= 0 || cols <= 0) return NK_OK;
  switch (kind) {
    case 0: return launch_cast<0>(in, rows, cols, ld_in, amax, out0, out1, ld_out, transpose, scale_out, st, sms, pro);
    case 1: return launch_cast<1>(in, rows, cols, ld_in, amax, out0, out1, ld_out, transpose, scale_out, st, sms, pro);
    case 2: return launch_cast<2>(in, rows, cols, ld_in, amax, out0, out1, ld_out, transpose, scale_out, st, sms, pro);
    default: return fail(NK_ERR_INVALID_ARG, "unknown cast kind %d", kind);
  }
}

nk_status ew_tensor(const float* x, const int64_t* sx, float* y, const int64_t* sy, const int64_t* shape, int rank,
                    const EwProg& prog, cudaStream_t st) {
  int sms = 0;
  nk_status s = require_device(&sms);
  if (s != NK_OK) return s;
  Strided4 g{};
  int64_t n = 1;
  for (int d = 0; d < 4; ++d) {
    const int src = d - (4 - rank);   // leading dimensions pad to extent 1
    g.shape[d] = src >= 0 ? shape[src] : 1;
    g.sx[d] = src >= 0 ? sx[src] : 0;
    g.sy[d] = src >= 0 ? sy[src] : 0;
    n *= g.shape[d];
  }
  if (n == 0) return NK_OK;
  // dense row-major X and Y with the same strides: one flat run
  bool dense = true;
  int64_t run = 1;
  for (int d = 3; d >= 0; --d) {
    if (g.shape[d] != 1 && (g.sx[d] != run || g.sy[d] != run)) dense = false;
    run *= g.shape[d];
  }
  const int64_t per = dense ? (n + 3) / 4 : n;
  int64_t blocks = (per + 255) / 256;
  if (blocks > (int64_t)sms * 16) blocks = (int64_t)sms * 16;
  if (blocks < 1) blocks = 1;
  const bool al = ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y)) & 15) == 0;
  if (dense && al) (void)nk::launch_k(ew_dense_kernel, dim3((unsigned)blocks), dim3(256), 0, st, 1, x, y, n, prog);
  else (void)nk::launch_k(ew_strided_kernel, dim3((unsigned)blocks), dim3(256), 0, st, 1, x, y, n, g, prog);
  return check_launch("elementwise kernel");
}

size_t norm_ws(int64_t, int64_t) { return 2 * kNormBlocks * sizeof(double); }

nk_status norm_sumsq(const float* C, int64_t ldc, const double* R, int64_t ldr, int64_t M,
                     int64_t N, double* out, void* ws, size_t ws_bytes, cudaStream_t st) {
  if (!ws || ws_bytes < norm_ws(M, N))
    return fail(NK_ERR_WORKSPACE, "norm needs %zu bytes of workspace", norm_ws(M, N));
  double* part = static_cast<double*>(ws);
  (void)nk::launch_k(norm_stage1, dim3(kNormBlocks), dim3(256), 0, st, 1, C, ldc, R, ldr, M, N, part);
  nk_status s = check_launch("norm_stage1");
  if (s != NK_OK) return s;
  (void)nk::launch_k(norm_stage2, dim3(1), dim3(1024), 0, st, 1, part, kNormBlocks, out);
  return check_launch("norm_stage2");
}

}  // namespace nk
