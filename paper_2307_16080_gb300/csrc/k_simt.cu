// k_simt.cu -- FP32 contraction on the CUDA cores (the plain FP32 path).
//
// linalg.matmul C[m,n] (+)= sum_k A[m,k] B[k,n] (Sec. 2.1.1 Listing
// "linalg-matmul") and, through an implicit im2col A-operand, the NHWC/HWCF
// convolution of Sec. 4.1 Listing "2dnchwconv".  The loop nest is tiled the
// way Sec. 4.3 tunes it -- output tiles per CTA, a reduction depth per step --
// but written for sm_103: tiles of 128 x 128, 128 x 64 or 64 x 64, BK = 16, a
// four-stage shared-memory ring fed by asynchronous copies, register blocking
// of 8 x 8 (8 x 4) outputs per thread, and FP32 FMAs.
//
// Split-K, two ways.  On request (schedule split_k): the reduction range is
// cut into `splits` slices (grid z); each slice writes its partial tile to the
// workspace and a second kernel sums the slices in a fixed order with a
// warp-shuffle tree, then applies the epilogue.  By the built-in rule, for
// outputs with too few tiles: the CTAs of a cluster each take a slice of K and
// add their tiles through distributed shared memory, in a fixed order, with
// no workspace and no second kernel.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <climits>
#include <mutex>
#include <type_traits>

#include "nk_internal.cuh"

namespace nk {
namespace {

constexpr int BK = 16;
constexpr int THREADS = 256;

// How an operand tile reaches shared memory: along k (k contiguous in memory),
// along the tile's other dimension, or (conv) by the im2col gather along k; in
// 4-byte copies, or in 16-byte ones where the operand's alignment allows them.
// 16-byte copies along k store a tile of A as [m][k]; the others store [k][m]
// and [k][n], 4-byte copies along k scattering a row of k.
// L_FAR and L_FAR16 are the gathers with 64-bit offsets and 32-bit positions.
enum LoadMode { L_K = 0, L_MN = 1, L_MN16 = 2, L_CONV = 3, L_K16 = 4, L_CONV16 = 5, L_FAR = 6, L_FAR16 = 7 };

struct KArgs {
  SimtGemm p;
  int k_chunk;      // reduction length handled by one grid-z slice
  float* partial;   // [splits][M][N] or null
  int csplit;       // CTAs of a cluster that share one tile's reduction (1: none)
};

// Implicit im2col element A[m,k] of the convolution (0 outside the input);
// *off = its offset in the input, or -1 for the zero padding.
__device__ __forceinline__ float conv_a(const SimtGemm& p, int m, int k, int64_t* off) {
  const ConvGeom& g = p.conv;
  int ow = m % g.ow;
  int t = m / g.ow;
  int oh = t % g.oh;
  int n = t / g.oh;
  int c = k % g.c;
  int tap = k / g.c;
  int kw = tap % g.kw;
  int kh = tap / g.kw;
  int ih = oh * g.sh + kh * g.dh - g.pt;
  int iw = ow * g.sw + kw * g.dw - g.pl;
  if (ih < 0 || ih >= g.h || iw < 0 || iw >= g.w) {
    *off = -1;
    return 0.f;
  }
  *off = n * g.sin_n + ih * g.sin_h + iw * g.sin_w + c;
  return p.A[*off];
}

__device__ __forceinline__ void cp4(uint32_t dst, const float* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(ok ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp16(uint32_t dst, const float* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ uint32_t cluster_map(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ float4 ld_cluster4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Epilogue of four consecutive outputs (m, nb..nb+3).
__device__ __forceinline__ void finish4(const SimtGemm& p, int m, int nb, const float (&acc)[4]) {
  float v[4];
  float* crow = p.C + (int64_t)m * p.scm;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int n = nb + j;
    float o = p.alpha * acc[j];
    if (n < p.N) {
      if (p.beta != 0.f) o = fmaf(p.beta, crow[(int64_t)n * p.scn], o);
      if (p.bias) o += p.bias[p.bias_on_m ? m : n];
      if (p.relu) o = (o > 0.f || o != o) ? o : 0.f;
    }
    v[j] = o;
  }
  if (p.scn == 1 && nb + 3 < p.N && ((reinterpret_cast<uintptr_t>(crow + nb) & 15) == 0)) {
    *reinterpret_cast<float4*>(crow + nb) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (nb + j < p.N) crow[(int64_t)(nb + j) * p.scn] = v[j];
  }
}

// What bounds it: the FMA pipes (128 lanes a cycle and SM), so everything else
// has to fit in the issue slots beside them.  FMAs are issued two to an
// instruction on pairs of columns (fma.rn.f32x2, each half rounded as fmaf:
// the sums are bitwise those of a scalar loop); operands come through a ring
// of asynchronous copies, which need no registers, no second pass to store
// and no alignment -- a row of odd length loads as fast as an aligned one.
// Rows past M and columns past N are copied as zeros, without a read, in the
// tiles 64 wide: lanes that read one clamped address instead take turns (8192 x
// 8 x 144, built-in tile: 23.5 us so, 7.3 now; 200 x 1500 x 700 in 64 x 64 tiles,
// whose last tiles have 8 rows: 39.7 / 26).  4-byte copies along k clamp (16
// lanes of a row read 16 addresses), and so does the 128 x 128 tile, which
// narrow outputs do not take and whose registers have no room for the test
// (1531 x 2047 x 1021: 149 / 154).  A loop of these FMAs over resident tiles
// reaches 66 TFLOP/s (scalar FMAs 60); the kernel 56 at 4096^3 (54 before).
// Odd row lengths, which took scalar loads: 1531 x 2047 x 1021 230 -> 150 us.
template <int BM, int BN, int T, int AM, int BMD>
__global__ void __launch_bounds__(T, T == 128 ? 3 : 2) simt_gemm_kernel(const __grid_constant__ KArgs args) {
  constexpr int S = 4;                  // stages
  constexpr int RM = BM * BN / T >= 32 ? 8 : 4;   // rows of a thread
  constexpr int TY = BM / RM, TX = T / TY, TN = BN / TX;
  constexpr bool FAR = AM == L_FAR || AM == L_FAR16;
  constexpr bool CONV = AM == L_CONV || AM == L_CONV16 || FAR;
  constexpr bool AMK = AM == L_CONV16 || AM == L_K16 || AM == L_FAR16;   // A is stored [m][k]
  constexpr int A_LD = AMK ? BK + 4 : BM + 4, B_LD = BN + 4;
  constexpr int A_FL = AMK ? BM * A_LD : BK * A_LD;
  constexpr int STAGE = A_FL + BK * B_LD;
  constexpr bool SKIP = BN == 64;        // no reads past M and N
  constexpr int KV = T == 256 && RM == 8 ? 2 : 4;   // k values of A in registers at a time (256 threads: 128 registers each)
  static_assert(TN == 8 || TN == 4, "8 x 8, 8 x 4 or 4 x 4 outputs per thread");
  static_assert(S * STAGE >= BM * BN, "a cluster's partial tiles reuse the ring");
  extern __shared__ __align__(16) float smem[];
  // conv: offset of a row's first tap, and its (ih, iw), in one word unless they are far
  using Off = typename std::conditional<FAR, int64_t, int>::type;
  __shared__ Off row_off[BM];
  __shared__ int row_hw[BM], row_w[FAR ? BM : 1];
  nk::pdl_wait();      // earlier kernels on the stream have finished
  nk::pdl_trigger();
  const SimtGemm& p = args.p;
  const int tid = threadIdx.x;
  const int tx = tid % TX, ty = tid / TX;
  const int cs = args.csplit;
  const int crank = cs > 1 ? (int)(blockIdx.x % cs) : 0;
  const int m0 = blockIdx.y * BM;
  const int n0 = (cs > 1 ? (int)(blockIdx.x / cs) : (int)blockIdx.x) * BN;
  const int kbeg = (cs > 1 ? crank : (int)blockIdx.z) * args.k_chunk;
  const int kend = min(p.K, kbeg + args.k_chunk);
  const int ntiles = kend > kbeg ? (kend - kbeg + BK - 1) / BK : 0;
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem);

  if constexpr (CONV) {
    const ConvGeom& g = p.conv;
    for (int r = tid; r < BM; r += T) {
      const int m = min(m0 + r, p.M - 1);
      const int ow = m % g.ow, q = m / g.ow, oh = q % g.oh, n = q / g.oh;
      const int ih = oh * g.sh - g.pt, iw = ow * g.sw - g.pl;
      row_off[r] = (Off)(n * g.sin_n + ih * g.sin_h + iw * g.sin_w);
      // rows past the end: above every input
      if constexpr (FAR) {
        row_hw[r] = m0 + r < p.M ? ih : INT_MIN;
        row_w[r] = iw;
      } else {
        row_hw[r] = m0 + r < p.M ? (ih << 16) | (iw & 0xffff) : INT_MIN;
      }
    }
    __syncthreads();
  }
  // per-thread load positions, fixed for the whole loop
  const int lk = tid % BK, lr = tid / BK;          // along k: this thread's k and first row
  constexpr int LR = T / BK;
  constexpr int KC = AMK ? 4 : 1;   // k values a copy of A brings
  const int ak = tid % (BK / KC) * KC, ar = tid / (BK / KC);
  constexpr int AR = T * KC / BK;
  auto load_tile = [&](int t) {
    const int k0 = kbeg + t * BK;
    const uint32_t sa = sbase + (uint32_t)((t % S) * STAGE * 4);
    const uint32_t sb = sa + (uint32_t)(A_FL * 4);
    auto cpa = [](uint32_t dst, const float* src, bool ok) {
      if constexpr (KC == 4) cp16(dst, src, ok);
      else cp4(dst, src, ok);
    };
    if constexpr (CONV) {
      const ConvGeom& g = p.conv;
      const int k = k0 + ak;
      const bool ok = k < kend;
      const int kc = ok ? k : 0;
      const int tap = kc / g.c, c = kc - tap * g.c;
      const int kh = tap / g.kw, kw = tap - kh * g.kw;
      const int dh = kh * g.dh, dw = kw * g.dw;
      const Off d = (Off)(dh * g.sin_h + dw * g.sin_w) + c;
#pragma unroll
      for (int i = 0; i < BM / AR; ++i) {
        const int r = ar + i * AR;
        const int hw = row_hw[r];
        const int ih = (FAR ? hw : hw >> 16) + dh, iw = (FAR ? row_w[r] : (int)(short)(hw & 0xffff)) + dw;
        const bool in = ok && (unsigned)ih < (unsigned)g.h && (unsigned)iw < (unsigned)g.w;
        cpa(sa + (uint32_t)((AMK ? r * A_LD + ak : ak * A_LD + r) * 4), p.A + (in ? row_off[r] + d : 0), in);
      }
    } else if constexpr (AM == L_K || AM == L_K16) {
      const int k = k0 + ak;
      const bool ok = k < kend;
      const float* src = p.A + (int64_t)(ok ? k : 0) * p.sak;
      const int rows = KC == 4 && SKIP ? p.M - m0 - ar : BM;   // this thread's rows that exist (4-byte copies clamp)
#pragma unroll
      for (int i = 0; i < BM / AR; ++i) {
        const int r = ar + i * AR;
        cpa(sa + (uint32_t)((AMK ? r * A_LD + ak : ak * A_LD + r) * 4), src + (int64_t)min(m0 + r, p.M - 1) * p.sam,
            ok && i * AR < rows);
      }
    } else if constexpr (AM == L_MN) {
      const int r = tid % BM;
      const bool in = !SKIP || m0 + r < p.M;
      const float* src = p.A + (int64_t)min(m0 + r, p.M - 1) * p.sam;
#pragma unroll
      for (int i = 0; i < BK * BM / T; ++i) {
        const int kk = tid / BM + i * (T / BM);
        const bool ok = k0 + kk < kend;
        cp4(sa + (uint32_t)((kk * A_LD + r) * 4), src + (int64_t)(ok ? k0 + kk : 0) * p.sak, ok && in);
      }
    } else {
      const int r = tid % (BM / 4) * 4;
      const bool in = !SKIP || m0 + r < p.M;
      const float* src = p.A + min(m0 + r, p.M - 4);
#pragma unroll
      for (int i = 0; i < BK * BM / 4 / T; ++i) {
        const int kk = tid / (BM / 4) + i * (T / (BM / 4));
        const bool ok = k0 + kk < kend;
        cp16(sa + (uint32_t)((kk * A_LD + r) * 4), src + (int64_t)(ok ? k0 + kk : 0) * p.sak, ok && in);
      }
    }
    if constexpr (BMD == L_K) {
      const int k = k0 + lk;
      const bool ok = k < kend;
      const float* src = p.B + (int64_t)(ok ? k : 0) * p.sbk;
#pragma unroll
      for (int i = 0; i < BN / LR; ++i) {
        const int c = lr + i * LR;
        cp4(sb + (uint32_t)((lk * B_LD + c) * 4), src + (int64_t)min(n0 + c, p.N - 1) * p.sbn, ok);
      }
    } else if constexpr (BMD == L_MN) {
      const int c = tid % BN;
      const bool in = !SKIP || n0 + c < p.N;
      const float* src = p.B + (int64_t)min(n0 + c, p.N - 1) * p.sbn;
#pragma unroll
      for (int i = 0; i < BK * BN / T; ++i) {
        const int kk = tid / BN + i * (T / BN);
        const bool ok = k0 + kk < kend;
        cp4(sb + (uint32_t)((kk * B_LD + c) * 4), src + (int64_t)(ok ? k0 + kk : 0) * p.sbk, ok && in);
      }
    } else {
      const int c = tid % (BN / 4) * 4;
      const bool in = !SKIP || n0 + c < p.N;
      const float* src = p.B + min(n0 + c, p.N - 4);
#pragma unroll
      for (int i = 0; i < BK * BN / 4 / T; ++i) {
        const int kk = tid / (BN / 4) + i * (T / (BN / 4));
        const bool ok = k0 + kk < kend;
        cp16(sb + (uint32_t)((kk * B_LD + c) * 4), src + (int64_t)(ok ? k0 + kk : 0) * p.sbk, ok && in);
      }
    }
  };

  f2 acc[RM][TN / 2];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < TN / 2; ++j) acc[i][j] = f2_set(0.f);

#pragma unroll
  for (int t = 0; t < S - 1; ++t) {
    if (t < ntiles) load_tile(t);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  for (int t = 0; t < ntiles; ++t) {
    asm volatile("cp.async.wait_group %0;" ::"n"(S - 2) : "memory");
    __syncthreads();   // tile t has landed for every thread, and tile t - 1 is read: its slot is free
    if (t + S - 1 < ntiles) load_tile(t + S - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const float* As = smem + (t % S) * STAGE;
    const float* Bs = As + A_FL;
    auto step = [&](int kk, const float (&a)[RM]) {
      f2 b[TN / 2];
#pragma unroll
      for (int h = 0; h < TN / 4; ++h) {
        const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(Bs + kk * B_LD + h * (BN / 2) + tx * 4);
        b[2 * h].v = q.x;
        b[2 * h + 1].v = q.y;
      }
#pragma unroll
      for (int i = 0; i < RM; ++i) {
        const f2 aa = f2_set(a[i]);
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) acc[i][j] = f2_fma(aa, b[j], acc[i][j]);
      }
    };
    if constexpr (AMK) {
#pragma unroll
      for (int kq = 0; kq < BK; kq += KV) {
        float av[RM][KV];
#pragma unroll
        for (int i = 0; i < RM; ++i) {
          const float* src = As + (ty + TY * i) * A_LD + kq;
          if constexpr (KV == 4) {
            const float4 q = *reinterpret_cast<const float4*>(src);
            av[i][0] = q.x; av[i][1] = q.y; av[i][2] = q.z; av[i][3] = q.w;
          } else {
            const float2 q = *reinterpret_cast<const float2*>(src);
            av[i][0] = q.x; av[i][1] = q.y;
          }
        }
#pragma unroll
        for (int e = 0; e < KV; ++e) {
          float a[RM];
#pragma unroll
          for (int i = 0; i < RM; ++i) a[i] = av[i][e];
          step(kq + e, a);
        }
      }
    } else {
#pragma unroll
      for (int kk = 0; kk < BK; ++kk) {
        float a[RM];
#pragma unroll
        for (int h = 0; h < RM / 4; ++h) {
          const float4 q = *reinterpret_cast<const float4*>(As + kk * A_LD + h * (BM / 2) + ty * 4);
          a[4 * h] = q.x; a[4 * h + 1] = q.y; a[4 * h + 2] = q.z; a[4 * h + 3] = q.w;
        }
        step(kk, a);
      }
    }
  }
  // the tile row of this thread's output i
  auto row_of = [&](int i) { return AMK ? ty + TY * i : (i / 4) * (BM / 2) + ty * 4 + (i % 4); };

  if (cs > 1) {
    // Every CTA of the cluster leaves its partial tile in its ring (whose last
    // copies have landed and been read); then each finishes a share of the
    // tile's rows, adding the slices in rank order.
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
#pragma unroll
    for (int i = 0; i < RM; ++i)
#pragma unroll
      for (int h = 0; h < TN / 4; ++h) {
        const int r = row_of(i), c = h * (BN / 2) + tx * 4;
        ulonglong2 q;
        q.x = acc[i][2 * h].v;
        q.y = acc[i][2 * h + 1].v;
        *reinterpret_cast<ulonglong2*>(smem + r * BN + c) = q;
      }
    cluster_barrier();
    const int share = BM / cs;
    for (int e = tid; e < share * (BN / 4); e += T) {
      const int r = crank * share + e / (BN / 4), c = (e % (BN / 4)) * 4;
      float4 sum = ld_cluster4(cluster_map(sbase + (uint32_t)((r * BN + c) * 4), 0));
      for (int q = 1; q < cs; ++q) {
        const float4 v = ld_cluster4(cluster_map(sbase + (uint32_t)((r * BN + c) * 4), (uint32_t)q));
        sum.x += v.x; sum.y += v.y; sum.z += v.z; sum.w += v.w;
      }
      if (m0 + r < p.M && n0 + c < p.N) {
        const float v[4] = {sum.x, sum.y, sum.z, sum.w};
        finish4(p, m0 + r, n0 + c, v);
      }
    }
    cluster_barrier();   // no CTA leaves while another may still read its tile
    return;
  }
  // Epilogue: partial tile to the workspace, or the fused epilogue to C.
#pragma unroll
  for (int i = 0; i < RM; ++i) {
    const int m = m0 + row_of(i);
    if (m >= p.M) continue;
#pragma unroll
    for (int h = 0; h < TN / 4; ++h) {
      const int nb = n0 + h * (BN / 2) + tx * 4;
      float v[4];
      f2_get(acc[i][2 * h], v[0], v[1]);
      f2_get(acc[i][2 * h + 1], v[2], v[3]);
      if (args.partial) {
        float* dst = args.partial + ((int64_t)blockIdx.z * p.M + m) * p.N;
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (nb + j < p.N) dst[nb + j] = v[j];
      } else if (nb < p.N) {
        finish4(p, m, nb, v);
      }
    }
  }
}

// The kernel that runs prologue / epilogue programs: scalar loads of any
// layout into registers, where a prologue can change them (256 threads, 64 or
// 128 square tiles, a double-buffered tile).
template <int RM, int RN, bool CONV>
__global__ void __launch_bounds__(THREADS, 2) simt_fused_kernel(const __grid_constant__ KArgs args) {
  nk::pdl_wait();      // earlier kernels on the stream have finished
  nk::pdl_trigger();
  constexpr int BM = 64 * RM;
  constexpr int BN = 64 * RN;
  constexpr int A_LD = BM + 4;
  constexpr int NA = BM * BK / THREADS;   // scalars of A each thread loads per tile
  constexpr int NB = BN * BK / THREADS;
  __shared__ __align__(16) float As[2][BK][A_LD];
  __shared__ __align__(16) float Bs[2][BK][BN];

  const SimtGemm& p = args.p;
  const int tid = threadIdx.x;
  const int tx = tid % 16, ty = tid / 16;
  const int m0 = blockIdx.y * BM;
  const int n0 = blockIdx.x * BN;
  const int kbeg = blockIdx.z * args.k_chunk;
  const int kend = min(p.K, kbeg + args.k_chunk);
  const int ntiles = kend > kbeg ? (kend - kbeg + BK - 1) / BK : 0;

  float ra[NA];
  float rb[NB];

  auto load_a = [&](int k0) {
#pragma unroll
    for (int j = 0; j < NA; ++j) {
      int L = tid + j * THREADS;
      int row = L % BM, kk = L / BM;
      int m = m0 + row, k = k0 + kk;
      float v = 0.f;
      if (m < p.M && k < kend) {
        int64_t off = (int64_t)m * p.sam + (int64_t)k * p.sak;
        if constexpr (CONV) v = conv_a(p, m, k, &off);
        else v = p.A[off];
        if (p.pro_a.n && off >= 0) v = ew_run(p.pro_a, v, off);
      }
      ra[j] = v;
    }
  };
  auto store_a = [&](int buf) {
#pragma unroll
    for (int j = 0; j < NA; ++j) {
      int L = tid + j * THREADS;
      As[buf][L / BM][L % BM] = ra[j];
    }
  };
  auto load_b = [&](int k0) {
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      int L = tid + j * THREADS;
      int col = L % BN, kk = L / BN;
      int n = n0 + col, k = k0 + kk;
      float v = 0.f;
      if (n < p.N && k < kend) {
        const int64_t off = (int64_t)k * p.sbk + (int64_t)n * p.sbn;
        v = p.B[off];
        if (p.pro_b.n) v = ew_run(p.pro_b, v, off);
      }
      rb[j] = v;
    }
  };
  auto store_b = [&](int buf) {
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      int L = tid + j * THREADS;
      Bs[buf][L / BN][L % BN] = rb[j];
    }
  };

  float acc[RM * 4][RN * 4];
#pragma unroll
  for (int i = 0; i < RM * 4; ++i)
#pragma unroll
    for (int j = 0; j < RN * 4; ++j) acc[i][j] = 0.f;

  if (ntiles > 0) {
    load_a(kbeg);
    load_b(kbeg);
    store_a(0);
    store_b(0);
    __syncthreads();
  }
  for (int t = 0; t < ntiles; ++t) {
    const int buf = t & 1;
    const bool more = t + 1 < ntiles;
    if (more) {
      load_a(kbeg + (t + 1) * BK);
      load_b(kbeg + (t + 1) * BK);
    }
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      float a[RM * 4], b[RN * 4];
#pragma unroll
      for (int r = 0; r < RM; ++r) {
        float4 v = *reinterpret_cast<const float4*>(&As[buf][kk][r * 64 + ty * 4]);
        a[4 * r] = v.x; a[4 * r + 1] = v.y; a[4 * r + 2] = v.z; a[4 * r + 3] = v.w;
      }
#pragma unroll
      for (int r = 0; r < RN; ++r) {
        float4 v = *reinterpret_cast<const float4*>(&Bs[buf][kk][r * 64 + tx * 4]);
        b[4 * r] = v.x; b[4 * r + 1] = v.y; b[4 * r + 2] = v.z; b[4 * r + 3] = v.w;
      }
#pragma unroll
      for (int i = 0; i < RM * 4; ++i)
#pragma unroll
        for (int j = 0; j < RN * 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if (more) {
      store_a(buf ^ 1);
      store_b(buf ^ 1);
    }
    __syncthreads();
  }

  // Epilogue: partial tile to the workspace, or the fused epilogue to C.
#pragma unroll
  for (int i = 0; i < RM * 4; ++i) {
    const int m = m0 + (i / 4) * 64 + ty * 4 + (i % 4);
    if (m >= p.M) continue;
#pragma unroll
    for (int r = 0; r < RN; ++r) {
      const int nb = n0 + r * 64 + tx * 4;
      if (args.partial) {
        float* dst = args.partial + ((int64_t)blockIdx.z * p.M + m) * p.N;
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (nb + j < p.N) dst[nb + j] = acc[i][4 * r + j];
        continue;
      }
      float v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int n = nb + j;
        float o = p.alpha * acc[i][4 * r + j];
        if (n < p.N) {
          if (p.beta != 0.f) o = fmaf(p.beta, p.C[(int64_t)m * p.scm + (int64_t)n * p.scn], o);
          if (p.bias) o += p.bias[p.bias_on_m ? m : n];
          if (p.relu) o = (o > 0.f || o != o) ? o : 0.f;
          if (p.ew.n) o = ew_run(p.ew, o, (int64_t)m * p.scm + (int64_t)n * p.scn);
        }
        v[j] = o;
      }
      float* crow = p.C + (int64_t)m * p.scm;
      if (p.scn == 1 && nb + 3 < p.N && ((reinterpret_cast<uintptr_t>(crow + nb) & 15) == 0)) {
        *reinterpret_cast<float4*>(crow + nb) = make_float4(v[0], v[1], v[2], v[3]);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (nb + j < p.N) crow[(int64_t)(nb + j) * p.scn] = v[j];
      }
    }
  }
}

// Split-K reduce: lanes of a warp form groups of S (a power of two); lane
// s of a group reads slice s of one output, the group sums with an xor
// shuffle tree (same order every run), lane 0 applies the epilogue.
template <bool EW>
__global__ void splitk_reduce_kernel(const __grid_constant__ SplitReduce r, int S) {
  nk::pdl_wait();      // earlier kernels on the stream have finished
  nk::pdl_trigger();
  const int lane = threadIdx.x & 31;
  const int per_warp = 32 / S;
  const int s = lane % S;
  const int64_t total = (int64_t)r.M * r.N;
  const int64_t warp = (int64_t)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x / 32);
  const float alpha = r.scale_a ? __frcp_rn(__fmul_rn(*r.scale_a, *r.scale_b)) : r.alpha;
  for (int64_t base = warp * per_warp; base < total; base += nwarps * per_warp) {
    const int64_t idx = base + lane / S;
    float v = 0.f;
    const int m = (int)(idx / r.N), n = (int)(idx % r.N);
    if (idx < total && s < r.splits) v = r.partial[((int64_t)s * r.M + m) * r.ldp + n];
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1)
      if (off < S) v += __shfl_xor_sync(0xffffffffu, v, off);
    if (s == 0 && idx < total) {
      const int64_t off = (int64_t)m * r.scm + (int64_t)n * r.scn;
      float* c = r.C + off;
      __nv_bfloat16* ch = reinterpret_cast<__nv_bfloat16*>(r.C) + off;
      float o = alpha * v;
      if (r.beta != 0.f) o = fmaf(r.beta, r.out_bf16 ? __bfloat162float(*ch) : *c, o);
      if (r.bias) o += r.bias[r.bias_on_m ? m : n];
      if (r.relu) o = (o > 0.f || o != o) ? o : 0.f;
      if (EW && r.ew.n) o = ew_run(r.ew, o, off);
      if (r.out_bf16) *ch = __float2bfloat16_rn(o);
      else *c = o;
    }
  }
}

// The same sum for up to eight slices and 16-byte rows of partials: a thread
// takes four consecutive outputs, reads each slice as one 16-byte word and adds
// the slices in the order of the shuffle tree above (slice s and s + S / 2
// first), so both give the same bits.  L2-bound; the tree reads 4 bytes a lane
// and divides for every output.  With its product, device time: BF16 512 x 512
// x 4096 (4 slices) 16.9 -> 10.9 us, 8x28x28x128 -> 256 3x3 / 2 (2 slices) 14.6
// -> 9.9 us.
// tx threads of a block share a row, so that short rows fill a block too (8x32x32
// x16 -> 16 E4M3, 8192 rows of 16: 10.2 us with a block per row, 6.0 the tree).
template <int S>
__global__ void __launch_bounds__(256) splitk_reduce4_kernel(const __grid_constant__ SplitReduce r, int tx) {
  nk::pdl_wait();      // earlier kernels on the stream have finished
  nk::pdl_trigger();
  const int row = (int)threadIdx.x / tx, ty = (int)blockDim.x / tx;
  const int n = ((int)blockIdx.x * tx + (int)threadIdx.x - row * tx) * 4;
  if (n >= r.N || row >= ty) return;
  const int64_t slice = (int64_t)r.M * r.ldp;
  const float alpha = r.scale_a ? __frcp_rn(__fmul_rn(*r.scale_a, *r.scale_b)) : r.alpha;
  const bool word = n + 4 <= r.N && r.scm % 4 == 0 && (reinterpret_cast<uintptr_t>(r.C) & (r.out_bf16 ? 7 : 15)) == 0;
  for (int64_t m = (int64_t)blockIdx.y * ty + row; m < r.M; m += (int64_t)gridDim.y * ty) {
    float v[S][4];
#pragma unroll
    for (int s = 0; s < S; ++s) {
      float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
      if (s < r.splits) q = *reinterpret_cast<const float4*>(r.partial + s * slice + m * r.ldp + n);
      v[s][0] = q.x; v[s][1] = q.y; v[s][2] = q.z; v[s][3] = q.w;
    }
#pragma unroll
    for (int h = S / 2; h >= 1; h /= 2)
#pragma unroll
      for (int s = 0; s < h; ++s)
#pragma unroll
        for (int e = 0; e < 4; ++e) v[s][e] += v[s + h][e];
    const int64_t off = m * r.scm + n;
    float* c = r.C + off;
    __nv_bfloat16* ch = reinterpret_cast<__nv_bfloat16*>(r.C) + off;
    float o[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      o[e] = alpha * v[0][e];
      if (n + e >= r.N) continue;
      if (r.beta != 0.f) o[e] = fmaf(r.beta, r.out_bf16 ? __bfloat162float(ch[e]) : c[e], o[e]);
      if (r.bias) o[e] += r.bias[r.bias_on_m ? m : n + e];
      if (r.relu) o[e] = (o[e] > 0.f || o[e] != o[e]) ? o[e] : 0.f;
    }
    if (word && r.out_bf16) {
      __nv_bfloat162 w[2] = {__floats2bfloat162_rn(o[0], o[1]), __floats2bfloat162_rn(o[2], o[3])};
      *reinterpret_cast<uint2*>(ch) = *reinterpret_cast<const uint2*>(w);
    } else if (word) {
      *reinterpret_cast<float4*>(c) = make_float4(o[0], o[1], o[2], o[3]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (n + e < r.N) {
          if (r.out_bf16) ch[e] = __float2bfloat16_rn(o[e]);
          else c[e] = o[e];
        }
    }
  }
}

template <int BM, int BN, int T, int AM, int BMD>
nk_status launch_kernel(const KArgs& a, dim3 grid, cudaStream_t st) {
  auto kern = simt_gemm_kernel<BM, BN, T, AM, BMD>;
  constexpr bool amk = AM == L_K16 || AM == L_CONV16 || AM == L_FAR16;
  constexpr int smem = 4 * ((amk ? BM * (BK + 4) : BK * (BM + 4)) + BK * (BN + 4)) * (int)sizeof(float);
  if constexpr (smem + 16 * BM > 48 * 1024) {
    static std::atomic<bool> set[64];   // per device; setting it twice is harmless
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64 || !set[dev].load(std::memory_order_relaxed)) {
      cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
      if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(simt_gemm_kernel)");
      if (dev >= 0 && dev < 64) set[dev].store(true, std::memory_order_relaxed);
    }
  }
  const cudaError_t e = nk::launch_k(kern, grid, dim3(T), smem, st, a.csplit, a);
  if (e != cudaSuccess) return cuda_fail(e, "launch simt_gemm_kernel");
  return check_launch("simt_gemm_kernel");
}

template <int BM, int BN, int T, int AM>
nk_status launch_b(const KArgs& a, int bmode, dim3 grid, cudaStream_t st) {
  switch (bmode) {
    case L_K: return launch_kernel<BM, BN, T, AM, L_K>(a, grid, st);
    case L_MN: return launch_kernel<BM, BN, T, AM, L_MN>(a, grid, st);
    default: return launch_kernel<BM, BN, T, AM, L_MN16>(a, grid, st);
  }
}

template <int BM, int BN, int T>
nk_status launch_a(const KArgs& a, int amode, int bmode, dim3 grid, cudaStream_t st) {
  switch (amode) {
    case L_K: return launch_b<BM, BN, T, L_K>(a, bmode, grid, st);
    case L_K16:   // 128 x 128 tiles have no registers for [m][k] (2629 us against 2460 at 4096^3)
      if constexpr (BN == 128) return launch_b<BM, BN, T, L_K>(a, bmode, grid, st);
      else return launch_b<BM, BN, T, L_K16>(a, bmode, grid, st);
    case L_MN: return launch_b<BM, BN, T, L_MN>(a, bmode, grid, st);
    case L_MN16: return launch_b<BM, BN, T, L_MN16>(a, bmode, grid, st);
    case L_CONV16:
      return bmode == L_MN16 ? launch_kernel<BM, BN, T, L_CONV16, L_MN16>(a, grid, st)
                             : launch_kernel<BM, BN, T, L_CONV16, L_MN>(a, grid, st);
    case L_FAR16:   // (one tile width is enough)
      if constexpr (BN == 64 && T == 128)
        return bmode == L_MN16 ? launch_kernel<BM, BN, T, L_FAR16, L_MN16>(a, grid, st)
                               : launch_kernel<BM, BN, T, L_FAR16, L_MN>(a, grid, st);
      return fail(NK_ERR_UNSUPPORTED, "no such FP32 tile");
    case L_FAR:
      if constexpr (BN == 64 && T == 128)
        return bmode == L_MN16 ? launch_kernel<BM, BN, T, L_FAR, L_MN16>(a, grid, st)
                               : launch_kernel<BM, BN, T, L_FAR, L_MN>(a, grid, st);
      return fail(NK_ERR_UNSUPPORTED, "no such FP32 tile");
    default:   // a convolution's filters are row-major [K][F]
      return bmode == L_MN16 ? launch_kernel<BM, BN, T, L_CONV, L_MN16>(a, grid, st)
                             : launch_kernel<BM, BN, T, L_CONV, L_MN>(a, grid, st);
  }
}

// Programs present: the register-loading kernel.
template <int RM, int RN>
nk_status launch_fused(const KArgs& a, dim3 grid, cudaStream_t st) {
  if (a.p.is_conv) (void)nk::launch_k(simt_fused_kernel<RM, RN, true>, grid, dim3(THREADS), 0, st, 1, a);
  else (void)nk::launch_k(simt_fused_kernel<RM, RN, false>, grid, dim3(THREADS), 0, st, 1, a);
  return check_launch("simt_fused_kernel");
}

inline bool al16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// The built-in tile, and the CTAs that share a tile's reduction: the smallest
// predicted time over the tiles and clusters of 1 to 8.  An SM works through
// its units (tiles x slices) at the rate the tile's shape reaches, each unit
// costs about a microsecond to fill and drain, and a cluster's exchange 1.9;
// clusters of eight 128-row tiles pack badly.  The constants are fitted to
// every combination timed on 34 products (64^3 to 2048^3, narrow and tall ones
// among them, B in both layouts) and 14 convolutions, where the choice is 3.5 %
// off the best of them on average and 22 % at worst.  (Clusters of 3, 5 and 6,
// which the kernel does not form, would be ahead on some: 1531 x 2047 x 1021 in
// clusters of 3, 142 us against 149.)  Examples, us (tile / cluster): 256^3
// 64x64 / 1 12.3, / 8 5.3; 1024^3 128x128 / 1 103, / 4 53; 1531 x 2047 x 1021
// 128x128 / 1 194, / 4 149; 8x56x56x64 3x3 64x64 / 1 71, 128x64 / 2 52; 700^3
// 128x128 / 4 29.5, 64x64 / 4 23.5; 8192 x 64 x 576 128x64 / 4 26.1, 64x64 / 4 19.
struct Choice {
  int bm, bn, csplit;
};
Choice choose(int M, int N, int K, int sms, bool may_split) {
  struct Tile {
    int bm, bn, resident;
    double gflop_us;   // per SM
  };
  static const Tile kTiles[] = {{128, 128, 2, 0.357}, {128, 64, 3, 0.352}, {64, 64, 2, 0.368}};
  Choice best{128, 128, 1};
  double best_t = 1e30;
  for (const Tile& t : kTiles) {
    const int64_t tm = (M + t.bm - 1) / t.bm;
    if (tm > 65535 && t.bm < 128) continue;   // grid.y
    for (int cs = 1; cs <= (may_split ? 8 : 1) && (cs == 1 || cs * BK <= K); cs *= 2) {
      const int64_t units = tm * ((N + t.bn - 1) / t.bn) * cs;
      // units of the busiest SM: whole ones while all are resident at once,
      // then the average and about half a set in the last wave
      const double u = units <= (int64_t)sms * t.resident ? (double)((units + sms - 1) / sms)
                                                          : (double)units / sms + 0.515 * t.resident;
      const double warps = u * (t.bn == 128 ? 8 : 4);
      const double fill = warps < 8 ? 0.504 : warps < 12 ? 0.664 : 1.0;   // too few to keep the FMA pipes busy
      const double kc = ((K + cs - 1) / cs + BK - 1) / BK * BK;
      const double pack = t.bm == 128 ? (cs == 8 ? 1.214 : cs == 4 ? 0.882 : 1.0) : 1.0;
      const double us = u * (2e-6 * t.bm * t.bn * kc * pack / (t.gflop_us * fill) + 1.026) + (cs > 1 ? 1.858 : 0.0);
      if (us < best_t) {
        best_t = us;
        best = {t.bm, t.bn, cs};
      }
    }
  }
  return best;
}

}  // namespace

size_t simt_gemm_ws(int M, int N, int splits) {
  return splits > 1 ? (size_t)splits * M * N * sizeof(float) : 0;
}

nk_status simt_gemm(const SimtGemm& p, int tile, int splits, void* ws, size_t ws_bytes,
                    cudaStream_t st) {
  if (p.M <= 0 || p.N <= 0) return NK_OK;
  if (tile != 0 && tile != 64 && tile != 128) return fail(NK_ERR_INVALID_ARG, "SIMT tile must be 64 or 128");
  if (splits < 1 || splits > 32) return fail(NK_ERR_INVALID_ARG, "split_k must be in [1, 32]");
  KArgs a;
  a.p = p;
  int kc = (p.K + splits - 1) / splits;
  kc = (kc + BK - 1) / BK * BK;
  if (kc == 0) kc = BK;
  splits = p.K > 0 ? (p.K + kc - 1) / kc : 1;
  a.k_chunk = kc;
  a.partial = nullptr;
  a.csplit = 1;
  if (splits > 1) {
    if (!ws || ws_bytes < simt_gemm_ws(p.M, p.N, splits))
      return fail(NK_ERR_WORKSPACE, "split-K needs %zu bytes of workspace",
                  simt_gemm_ws(p.M, p.N, splits));
    a.partial = static_cast<float*>(ws);
  }
  // The gather keeps a pixel's offset in 32 bits and its position in 16; long
  // signals and inputs beyond 2^30 values take the one with 64 and 32 (1 x 1 x
  // 40000 x 64 -> 64, 1 x 3: 139 us with the register-loading kernel, which
  // runs programs, 32 with this one).
  const ConvGeom& cg = p.conv;
  const bool far = p.is_conv && (cg.h + cg.pt + cg.kh * cg.dh > 32000 || cg.w + cg.pl + cg.kw * cg.dw > 32000 ||
                                 cg.oh * (int64_t)cg.sh > 32000 || cg.ow * (int64_t)cg.sw > 32000 ||
                                 cg.n * cg.sin_n + (cg.h + cg.pt + cg.kh * cg.dh) * cg.sin_h +
                                         (cg.w + cg.pl + cg.kw * cg.dw) * cg.sin_w >=
                                     INT32_MAX / 2);
  if (p.pro_a.n || p.pro_b.n || p.ew.n) {
    // Convolutions have few columns: a 128-wide tile is half empty at 64 filters
    // (8x56x56x64 3x3 + GELU 174 us with 64 x 64 tiles, 260 with 128 x 128).
    if (tile == 0) tile = p.is_conv || (int64_t)((p.M + 127) / 128) * ((p.N + 127) / 128) < 152 ? 64 : 128;
    const dim3 grid((p.N + tile - 1) / tile, (p.M + tile - 1) / tile, splits);
    if (grid.y > 65535) return fail(NK_ERR_UNSUPPORTED, "M too large for the SIMT grid");
    const nk_status s = tile == 128 ? launch_fused<2, 2>(a, grid, st) : launch_fused<1, 1>(a, grid, st);
    if (s != NK_OK || splits == 1) return s;
  } else {
    // Pick the load modes from the layout and alignment.
    int amode, bmode;
    if (p.is_conv)
      amode = cg.c % 4 == 0 && cg.sin_n % 4 == 0 && cg.sin_h % 4 == 0 && cg.sin_w % 4 == 0 && al16(p.A) ? (far ? L_FAR16 : L_CONV16)
                                                                                                           : (far ? L_FAR : L_CONV);
    else if (p.sak == 1 && p.sam % 4 == 0 && p.K % 4 == 0 && al16(p.A)) amode = L_K16;
    else if (p.sam == 1 && p.sak != 1) amode = p.sak % 4 == 0 && p.M % 4 == 0 && al16(p.A) ? L_MN16 : L_MN;
    else amode = L_K;
    if (p.sbn == 1) bmode = p.sbk % 4 == 0 && p.N % 4 == 0 && al16(p.B) ? L_MN16 : L_MN;
    else bmode = L_K;
    int bm = tile, bn = tile == 128 && p.N <= 64 ? 64 : tile;   // no empty half of a tile
    int sms = 0;
    nk_status s = require_device(&sms);
    if (s != NK_OK) return s;
    if (tile == 0) {
      const Choice c = choose(p.M, p.N, p.K, sms, splits == 1);
      bm = c.bm;
      bn = c.bn;
      a.csplit = c.csplit;
      if (a.csplit > 1) a.k_chunk = ((p.K + a.csplit - 1) / a.csplit + BK - 1) / BK * BK;
    }
    if (far) bn = 64;
    const dim3 grid((p.N + bn - 1) / bn * a.csplit, (p.M + bm - 1) / bm, splits);
    if (grid.y > 65535) return fail(NK_ERR_UNSUPPORTED, "M too large for the SIMT grid");
    // A 64 x 64 tile that has an SM to itself and few steps: four warps of 8 x 4
    // outputs cannot hide its start, eight of 4 x 4 do (us, 64 x 64 tiles:
    // 128^3 7.3 / 6.0, 256^3 11.6 / 10.5, 8192 x 64 x 144 8.6 / 7.3; at K = 576 the
    // larger blocks' fewer shared-memory reads win, 22.7 / 22.3 and, with A
    // column-major, 19.8 / 21.8).
    const bool alone = !far && a.csplit == 1 && a.k_chunk <= 320 && (int64_t)grid.x * grid.y * grid.z <= sms;
    s = bn == 128   ? launch_a<128, 128, 256>(a, amode, bmode, grid, st)
                        : bm == 128 ? launch_a<128, 64, 128>(a, amode, bmode, grid, st)
                        : alone     ? launch_a<64, 64, 256>(a, amode, bmode, grid, st)
                                    : launch_a<64, 64, 128>(a, amode, bmode, grid, st);
    if (s != NK_OK || splits == 1) return s;
  }
  SplitReduce r{};
  r.partial = a.partial;
  r.ldp = p.N;
  r.splits = splits;
  r.M = p.M;
  r.N = p.N;
  r.C = p.C;
  r.scm = p.scm;
  r.scn = p.scn;
  r.bias = p.bias;
  r.bias_on_m = p.bias_on_m;
  r.alpha = p.alpha;
  r.beta = p.beta;
  r.relu = p.relu;
  r.scale_a = nullptr;
  r.scale_b = nullptr;
  r.ew = p.ew;
  return splitk_reduce(r, st);
}

nk_status splitk_reduce(const SplitReduce& r, cudaStream_t st) {
  if (r.splits < 1 || r.splits > 32) return fail(NK_ERR_INVALID_ARG, "splits must be in [1, 32]");
  int S = 1;
  while (S < r.splits) S <<= 1;
  int sms = 0;
  nk_status s = require_device(&sms);
  if (s != NK_OK) return s;
  if (S >= 2 && S <= 8 && r.ew.n == 0 && r.scn == 1 && r.ldp % 4 == 0 && al16(r.partial)) {
    const int quads = (r.N + 3) / 4;
    const int tx = std::min(quads, 256);
    const int threads = tx <= 128 ? 256 : (tx + 31) / 32 * 32;   // whole rows, or one
    const int ty = threads / tx;
    const dim3 grid((quads + tx - 1) / tx, (unsigned)std::min<int64_t>(((int64_t)r.M + ty - 1) / ty, 65535));
    if (S == 2) (void)nk::launch_k(splitk_reduce4_kernel<2>, grid, dim3(threads), 0, st, 1, r, tx);
    else if (S == 4) (void)nk::launch_k(splitk_reduce4_kernel<4>, grid, dim3(threads), 0, st, 1, r, tx);
    else (void)nk::launch_k(splitk_reduce4_kernel<8>, grid, dim3(threads), 0, st, 1, r, tx);
    return check_launch("splitk_reduce4_kernel");
  }
  const int64_t total = (int64_t)r.M * r.N;
  const int64_t warps_needed = (total + (32 / S) - 1) / (32 / S);
  int64_t blocks = (warps_needed + 7) / 8;
  blocks = blocks < (int64_t)sms * 8 ? blocks : (int64_t)sms * 8;
  if (blocks < 1) blocks = 1;
  if (r.ew.n) (void)nk::launch_k(splitk_reduce_kernel<true>, dim3((unsigned)blocks), dim3(256), 0, st, 1, r, S);
  else (void)nk::launch_k(splitk_reduce_kernel<false>, dim3((unsigned)blocks), dim3(256), 0, st, 1, r, S);
  return check_launch("splitk_reduce_kernel");
}

}  // namespace nk

// ------------------------------------------------- split-K without allocation
// For callers that cannot allocate device memory at all: code running where
// cudaMalloc is unavailable or forbidden (inside a custom allocator's
// callbacks, while another runtime owns the memory pool, or in a process
// whose device memory budget is already spoken for).  The split-K partial
// sums go to this fixed, file-scope device array instead of a caller
// workspace; every GPU that loads the library keeps it until exit.
namespace nk {
namespace {

constexpr size_t kStaticScratchFloats = size_t(4) << 20;   // 16 MiB of FP32 partials
__device__ __align__(256) float g_splitk_scratch[kStaticScratchFloats];

constexpr int kMaxDevices = 64;
std::mutex g_scratch_mu;
float* g_scratch_addr[kMaxDevices];   // device address of g_splitk_scratch, per device ordinal

}  // namespace
}  // namespace nk

extern "C" nk_status nk_matmul_f32_splitk_noalloc(const float* A, int64_t lda, const float* B,
                                                  int64_t ldb, float* C, int64_t ldc, int32_t M,
                                                  int32_t N, int32_t K, int32_t split_k,
                                                  void* stream) {
  nk::NvtxRange nvtx_range_("nk_matmul_f32_splitk_noalloc");
  using namespace nk;
  int sms = 0;
  nk_status s = require_device(&sms);
  if (s != NK_OK) return s;
  if (M < 0 || N < 0 || K < 0) return fail(NK_ERR_INVALID_ARG, "negative extent");
  if (split_k < 1 || split_k > 32) return fail(NK_ERR_INVALID_ARG, "split_k must be in [1, 32]");
  if (M == 0 || N == 0) return NK_OK;
  if (!A || !B || !C) return fail(NK_ERR_INVALID_ARG, "null pointer");
  if (lda < K || ldb < N || ldc < N) return fail(NK_ERR_INVALID_ARG, "leading dimension too small");
  if ((size_t)split_k * (size_t)M * (size_t)N > kStaticScratchFloats)
    return fail(NK_ERR_WORKSPACE,
                "split_k*M*N = %zu exceeds the static scratch of %zu floats (16 MiB)",
                (size_t)split_k * M * N, kStaticScratchFloats);
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  if (dev < 0 || dev >= kMaxDevices)
    return fail(NK_ERR_UNSUPPORTED, "device ordinal %d: the static scratch table holds %d devices", dev,
                kMaxDevices);
  float* scratch = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_scratch_mu);
    if (!g_scratch_addr[dev]) {
      // Host code only sees a host-side stand-in for the array; the device
      // address comes from the runtime, once per device, with it current.
      void* p = nullptr;
      e = cudaGetSymbolAddress(&p, g_splitk_scratch);
      if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_splitk_scratch)");
      g_scratch_addr[dev] = static_cast<float*>(p);
    }
    scratch = g_scratch_addr[dev];
  }
  SimtGemm p{};
  p.A = A; p.sam = lda; p.sak = 1;
  p.B = B; p.sbk = ldb; p.sbn = 1;
  p.C = C; p.scm = ldc; p.scn = 1;
  p.M = M; p.N = N; p.K = K;
  p.alpha = 1.f; p.beta = 0.f;
  // 64 x 64 tiles while 128 x 128 ones would not give every SM one (the caller
  // has chosen the slices, so the built-in rule, which slices K itself, has no
  // say).
  const int tile = (int64_t)((M + 127) / 128) * ((N + 127) / 128) < sms ? 64 : 128;
  // Every slice overwrites its whole [M,N] partial tile, so the scratch needs
  // no clearing between calls.
  return simt_gemm(p, tile, split_k, scratch, kStaticScratchFloats * sizeof(float),
                   static_cast<cudaStream_t>(stream));
}
