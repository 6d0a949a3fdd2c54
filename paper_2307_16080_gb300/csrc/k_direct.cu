// k_direct.cu -- the convolution of Sec. 4.1 Listing "2dnchwconv" as written:
// NCHW input, FCHW kernel, output-parallel,
//   out[n,co,ho,wo] += in[n, ci, ho*sh + ki*dh - pt, wo*sw + kj*dw - pl] * ker[co,ci,ki,kj]
// (stride 1, no padding in the listing; stride, dilation and zero padding
// here).  With a handful of channels -- the tuning experiment of Sec. 4.3
// uses (N, C, H, W) = (1, 1, 1280, 1280) and (Ci, Co, K) = (1, 3, 3) -- the
// contraction is far too short for tensor cores and the kernel is bound by
// HBM: each input element is read once through a shared-memory halo tile,
// each output element written once with 128-bit stores.
//
// Three kernels:
//   direct_rows_kernel (stride 1, dilation 1, 1x1 / 3x3 / 5x5 filters): each
//     thread owns 4 consecutive output columns of ROWS consecutive rows for
//     up to four output channels and walks down the ROWS + KH - 1 input rows
//     it needs, one register segment of 4 + KW - 1 values per row (each input
//     row feeds every output row and tap that uses it), so the input is read
//     from DRAM once, with no shared memory; the filter taps of an input
//     channel sit in registers.  Outputs leave as 16-byte stores (8-byte or
//     single ones on rows that are not aligned to them).
//   direct_stream_kernel (1x1 to one output channel and 3x3 filters, one input
//     channel -- the tuning experiment's Ci = 1 -- on large images): as above,
//     but a thread walks `rpt` output rows keeping only KH rotating accumulator
//     rows; an output row is stored as soon as its last tap row has arrived, so
//     the halo rows are amortised over many rows and the stores spread through
//     the loop.
//   direct_conv_kernel (any stride / dilation / filter up to 64 taps): a CTA
//     computes a 16 x 64 output tile of one image for up to 8 output
//     channels from a halo tile staged in shared memory, one input channel
//     at a time.
#include <cuda_runtime.h>

#include "nk_internal.cuh"

namespace nk {
namespace {

constexpr int TH = 16, TW = 64, CO_G = 8, THREADS = 256;
constexpr int MAX_IN_H = 64, MAX_IN_W = 176;   // halo tile limits (44 KB of shared memory)

struct Direct {
  const float* I;
  int64_t sIn, sIc, sIh;   // input strides (width stride 1)
  const float* Kr;         // FCHW, contiguous
  float* O;
  int64_t sOn, sOc, sOh;   // output strides (width stride 1)
  int N, CI, H, W, CO, KH, KW, OH, OW;
  int sh, sw, dh, dw, pt, pl;
  const float* bias;
  int relu;
  float beta;
  int in_h, in_w;          // halo tile extent
  EwProg ew;               // fused elementwise program (offsets from O)
};

// Shared memory is sized to the actual halo tile (18 x 66 floats for a 3 x 3
// stride-1 filter), so many CTAs share an SM and keep enough loads in flight
// to reach HBM bandwidth.
__global__ void __launch_bounds__(THREADS) direct_conv_kernel(const __grid_constant__ Direct p) {
  nk::pdl_wait();      // earlier kernels on the stream have finished
  nk::pdl_trigger();
  extern __shared__ float smem_f[];
  float* ker = smem_f;                    // [CO_G][64] taps of one input channel
  float* tile = smem_f + CO_G * 64;       // [in_h][in_w] halo tile
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  const int wo0 = blockIdx.x * TW, ho0 = blockIdx.y * TH;
  const int n = blockIdx.z / ((p.CO + CO_G - 1) / CO_G);
  const int cg = blockIdx.z % ((p.CO + CO_G - 1) / CO_G);
  const int co0 = cg * CO_G;
  const int ncog = min(CO_G, p.CO - co0);
  const int ho = ho0 + ty;
  const int wo = wo0 + tx * 4;
  const int taps = p.KH * p.KW;
  const int ih0 = ho0 * p.sh - p.pt, iw0 = wo0 * p.sw - p.pl;
  float acc[CO_G][4];
#pragma unroll
  for (int c = 0; c < CO_G; ++c)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[c][j] = 0.f;

  for (int ci = 0; ci < p.CI; ++ci) {
    __syncthreads();
    const float* src = p.I + n * p.sIn + ci * p.sIc;
    for (int e = threadIdx.x; e < ncog * taps; e += THREADS) {
      const int c = e / taps, t = e % taps;
      ker[c * 64 + t] = p.Kr[((int64_t)(co0 + c) * p.CI + ci) * taps + t];
    }
    // Eight loads in flight per thread before any lands in shared memory.
    const int total = p.in_h * p.in_w;
    for (int e0 = threadIdx.x; e0 < total; e0 += 8 * THREADS) {
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int e = e0 + u * THREADS;
        const int r = e / p.in_w, c = e - r * p.in_w;
        const int ih = ih0 + r, iw = iw0 + c;
        v[u] = (e < total && ih >= 0 && ih < p.H && iw >= 0 && iw < p.W) ? src[ih * p.sIh + iw] : 0.f;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (e0 + u * THREADS < total) tile[e0 + u * THREADS] = v[u];
    }
    __syncthreads();
    for (int ki = 0; ki < p.KH; ++ki) {
      const int r = ty * p.sh + ki * p.dh;
      for (int kj = 0; kj < p.KW; ++kj) {
        float x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) x[j] = tile[r * p.in_w + (tx * 4 + j) * p.sw + kj * p.dw];
        const int t = ki * p.KW + kj;
#pragma unroll
        for (int c = 0; c < CO_G; ++c) {
          if (c < ncog) {
            const float w = ker[c * 64 + t];
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[c][j] = fmaf(x[j], w, acc[c][j]);
          }
        }
      }
    }
  }
  if (ho >= p.OH) return;
#pragma unroll
  for (int c = 0; c < CO_G; ++c) {
    if (c >= ncog) break;
    float* dst = p.O + n * p.sOn + (int64_t)(co0 + c) * p.sOc + (int64_t)ho * p.sOh + wo;
    const float b = p.bias ? p.bias[co0 + c] : 0.f;
    float v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float o = acc[c][j];
      if (p.beta != 0.f && wo + j < p.OW) o = fmaf(p.beta, dst[j], o);
      o += b;
      if (p.relu) o = (o > 0.f || o != o) ? o : 0.f;
      if (p.ew.n && wo + j < p.OW) o = ew_run(p.ew, o, (dst - p.O) + j);
      v[j] = o;
    }
    if (wo + 3 < p.OW && ((reinterpret_cast<uintptr_t>(dst) & 15) == 0)) {
      *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (wo + j < p.OW) dst[j] = v[j];
    }
  }
}

// Input segment x[0..SEG) of a row that starts at src; wi is the column of
// src[0], columns outside [0, W) are zero.  vec: the whole warp's segments are
// 16-byte aligned and inside the row.
template <int SEG>
__device__ __forceinline__ void load_row(const float* src, bool vec, int wi, int W, float (&x)[SEG]) {
  if (SEG >= 4 && vec) {
    const float4 v = *reinterpret_cast<const float4*>(src);
    x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
    if constexpr (SEG == 6) {
      const float2 t = *reinterpret_cast<const float2*>(src + 4);
      x[4] = t.x; x[5] = t.y;
    } else if constexpr (SEG == 8) {
      const float4 t = *reinterpret_cast<const float4*>(src + 4);
      x[4] = t.x; x[5] = t.y; x[6] = t.z; x[7] = t.w;
    }
  } else {
#pragma unroll
    for (int j = 0; j < SEG; ++j) x[j] = (unsigned)(wi + j) < (unsigned)W ? src[j] : 0.f;
  }
}

// Epilogue and store of a lane's four outputs at d, on a row that starts s
// floats before a 16-byte boundary; full: every lane of the warp has all four.
template <bool PLAIN>
__device__ __forceinline__ void finish_row(const Direct& p, float* d, int s, bool full, int wo, float bias,
                                           const float (&acc)[4]) {
  float v[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float o = acc[j];
    if constexpr (!PLAIN)
      if (p.beta != 0.f && wo + j < p.OW) o = fmaf(p.beta, d[j], o);
    o += bias;
    if constexpr (!PLAIN)
      if (p.relu) o = (o > 0.f || o != o) ? o : 0.f;
    v[j] = o;
  }
  if (full && s == 0) {
    *reinterpret_cast<float4*>(d) = make_float4(v[0], v[1], v[2], v[3]);
  } else if (full && s == 2) {
    *reinterpret_cast<float2*>(d) = make_float2(v[0], v[1]);
    *reinterpret_cast<float2*>(d + 2) = make_float2(v[2], v[3]);
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (full || wo + j < p.OW) d[j] = v[j];
  }
}

// CTAs per SM that direct_rows_kernel's registers have to leave room for: its
// loads are hidden by other warps alone.  16 x 3 x 1280 x 1280 -> 3, 3 x 3: 219 us
// at seven CTAs, 286 with the registers the compiler would take; 16 x 3 x 700 x
// 800 -> 4, 5 x 5 in pairs of channels: 162 at eight, 176 at six; 8 x 3 x 640 x 640
// -> 3, 5 x 5: 57 at four, 72 at five (spills).
constexpr int rows_ctas(int kh, int co) {
  return kh == 5 ? (co == 1 ? 10 : co == 2 ? 8 : 4)
       : kh == 3 ? (co == 1 ? 12 : co == 2 ? 9 : co == 3 ? 7 : 5)
                 : (co <= 2 ? 16 : co == 3 ? 12 : 9);
}

// Blocks of rows: a thread owns four columns of ROWS output rows and walks the
// ROWS + KH - 1 input rows of one channel after another.  Issue slots bound it
// like the kernel below, so it has the same exact CO, PLAIN, and alignment
// settled once.
template <int KH, int KW, int CO, int ROWS, bool PLAIN>
__global__ void __launch_bounds__(128, rows_ctas(KH, CO)) direct_rows_kernel(const __grid_constant__ Direct p, int cols) {
  nk::pdl_wait();      // earlier kernels on the stream have finished
  nk::pdl_trigger();
  constexpr int SEG = 4 + KW - 1;
  constexpr int TAPS = KH * KW;
  const int lane = threadIdx.x & 31;
  const int by = blockIdx.x / cols;   // grid.x: `cols` blocks of columns for each block of rows
  const int wo = (blockIdx.x - by * cols) * 512 + threadIdx.x * 4;   // first of this thread's 4 output columns
  const int ho0 = by * ROWS;
  const int groups = (p.CO + CO - 1) / CO;
  const int n = blockIdx.y / groups;
  const int co0 = (blockIdx.y % groups) * CO;
  const int ncog = min(CO, p.CO - co0);
  if (wo - lane * 4 >= p.OW) return;   // whole warps: the votes below ask every lane
  float acc[ROWS][CO][4];
#pragma unroll
  for (int r = 0; r < ROWS; ++r)
#pragma unroll
    for (int c = 0; c < CO; ++c)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[r][c][j] = 0.f;
  const float* src = p.I + n * p.sIn + (int64_t)(ho0 - p.pt) * p.sIh + (wo - p.pl);
  const bool vec = __all_sync(0xffffffffu, wo - p.pl >= 0 && wo - p.pl + SEG <= p.W && (p.sIh & 3) == 0 &&
                                               ((p.sIc & 3) == 0 || p.CI == 1) &&
                                               (reinterpret_cast<uintptr_t>(src) & 15) == 0);
#pragma unroll 1
  for (int ci = 0; ci < p.CI; ++ci, src += p.sIc) {
    float w[CO][TAPS];
#pragma unroll
    for (int c = 0; c < CO; ++c)
#pragma unroll
      for (int t = 0; t < TAPS; ++t)
        w[c][t] = c < ncog ? p.Kr[((int64_t)(co0 + c) * p.CI + ci) * TAPS + t] : 0.f;
#pragma unroll
    for (int r = 0; r < ROWS + KH - 1; ++r) {   // input row ho0 + r - pt
      float x[SEG];
      const int ih = ho0 + r - p.pt;
      if ((unsigned)ih < (unsigned)p.H) {
        load_row<SEG>(src + (int64_t)r * p.sIh, vec, wo - p.pl, p.W, x);
      } else {
#pragma unroll
        for (int j = 0; j < SEG; ++j) x[j] = 0.f;
      }
#pragma unroll
      for (int kh = 0; kh < KH; ++kh) {
        const int orow = r - kh;   // the output row this input row meets through tap row kh
        if (orow < 0 || orow >= ROWS) continue;
#pragma unroll
        for (int c = 0; c < CO; ++c)
#pragma unroll
          for (int kw = 0; kw < KW; ++kw)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[orow][c][j] = fmaf(x[j + kw], w[c][kh * KW + kw], acc[orow][c][j]);
      }
    }
  }
  const bool full = __all_sync(0xffffffffu, wo + 3 < p.OW);
  float* dst = p.O + n * p.sOn + (int64_t)co0 * p.sOc + (int64_t)ho0 * p.sOh + wo;
  // floats into a 16-byte word at which a row starts: wo is a multiple of 4
  const int at = (int)((reinterpret_cast<uintptr_t>(p.O) >> 2) + n * p.sOn + co0 * p.sOc + ho0 * p.sOh);
  float bias[CO];   // read before the first store, which the compiler cannot move it across
#pragma unroll
  for (int c = 0; c < CO; ++c) bias[c] = (p.bias && c < ncog) ? p.bias[co0 + c] : 0.f;
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    if (ho0 + r >= p.OH) break;
#pragma unroll
    for (int c = 0; c < CO; ++c) {
      if (c >= ncog) break;
      const int s = -(at + c * (int)(p.sOc & 3) + r * (int)(p.sOh & 3)) & 3;
      finish_row<PLAIN>(p, dst + c * p.sOc + r * p.sOh, s, full, wo, bias[c], acc[r][c]);
    }
  }
}

// One input channel: output row o lives in accumulator slot o % KH while
// input rows o .. o+KH-1 arrive; it is stored after the last of them.  The
// next input row's loads are in flight while a row is used.
//
// What bounds it is issue slots, not HBM (an input row feeds KH x KW x CO FMAs
// per output column, beside the loads' and stores' bookkeeping), so CO is the
// exact number of output channels of the thread, PLAIN leaves accumulate and
// ReLU out, and range and alignment are settled once per thread where they can
// be.  16 x 1280 x 1280, 3 x 3, 1 -> 3 channels (418 MB): 330 instructions per
// warp and row, four channels computed for three and 8-byte stores on every
// other row took 123 us; now 69 us, 90 % of the copy rate.  Rows on odd floats: single stores; putting
// two lanes' values together into aligned 16-byte ones costs more issue slots
// than it saves (16 x 1000 x 1001 1 -> 4, 3 x 3: 91 us so, 68 us now).
template <int KH, int KW, int CO, bool PLAIN>
__global__ void __launch_bounds__(128) direct_stream_kernel(const __grid_constant__ Direct p, int rpt) {
  nk::pdl_wait();      // earlier kernels on the stream have finished
  nk::pdl_trigger();
  constexpr int SEG = 4 + KW - 1;
  constexpr int TAPS = KH * KW;
  const int lane = threadIdx.x & 31;
  const int wo = blockIdx.x * 512 + threadIdx.x * 4;
  const int ho0 = blockIdx.y * rpt;
  const int groups = (p.CO + CO - 1) / CO;
  const int n = blockIdx.z / groups;
  const int co0 = (blockIdx.z % groups) * CO;
  const int ncog = min(CO, p.CO - co0);
  if (wo - lane * 4 >= p.OW || ho0 >= p.OH) return;   // whole warps: the votes below ask every lane
  const int rows = min(rpt, p.OH - ho0);
  float w[CO][TAPS];
#pragma unroll
  for (int c = 0; c < CO; ++c)
#pragma unroll
    for (int t = 0; t < TAPS; ++t) w[c][t] = c < ncog ? p.Kr[(int64_t)(co0 + c) * TAPS + t] : 0.f;
  float bias[CO];
#pragma unroll
  for (int c = 0; c < CO; ++c) bias[c] = (p.bias && c < ncog) ? p.bias[co0 + c] : 0.f;
  // Accumulators of the KH output rows under way.  A row's first tap row
  // overwrites its slot, so the rows above the first output row (o < 0) leave
  // nothing behind, and those past the last are never stored.
  float acc[KH][CO][4];
#pragma unroll
  for (int i = 0; i < KH; ++i)
#pragma unroll
    for (int c = 0; c < CO; ++c)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][c][j] = 0.f;
  const int nin = rows + KH - 1;   // input rows ho0 - pt .. ho0 - pt + nin - 1
  const float* src = p.I + n * p.sIn + (int64_t)(ho0 - p.pt) * p.sIh + (wo - p.pl);   // next row to load
  float* dst = p.O + n * p.sOn + (int64_t)co0 * p.sOc + (int64_t)ho0 * p.sOh + wo;
  // settled once, for whole warps: every lane's loads are aligned and inside
  // the row, every lane's four outputs exist; floats from a row to the next
  // 16-byte boundary (the same for every lane: wo is a multiple of 4)
  const bool vec = __all_sync(0xffffffffu, wo - p.pl >= 0 && wo - p.pl + SEG <= p.W && (p.sIh & 3) == 0 &&
                                               (reinterpret_cast<uintptr_t>(src) & 15) == 0);
  const bool full = __all_sync(0xffffffffu, wo + 3 < p.OW);
  const int sOc4 = (int)(p.sOc & 3), sOh4 = (int)(p.sOh & 3);
  int at = (int)((reinterpret_cast<uintptr_t>(p.O) >> 2) + n * p.sOn + co0 * p.sOc + ho0 * p.sOh);
  auto load = [&](int r, float (&x)[SEG]) {
    const int ih = ho0 + r - p.pt;
    if (r < nin && ih >= 0 && ih < p.H) {
      load_row<SEG>(src, vec, wo - p.pl, p.W, x);
    } else {
#pragma unroll
      for (int j = 0; j < SEG; ++j) x[j] = 0.f;
    }
    src += p.sIh;
  };
  constexpr int U = KH == 1 ? 4 : KH;   // rows in flight, and unrolled: buffers and slots are compile-time
  float nx[U][SEG];
#pragma unroll
  for (int u = 0; u < U; ++u) load(u, nx[u]);
#pragma unroll 1
  for (int r0 = 0; r0 < nin; r0 += U) {
#pragma unroll
    for (int u = 0; u < U; ++u) {   // input row r = r0 + u, r0 a multiple of U (and so of KH)
      const int r = r0 + u;
      if (r >= nin) break;
      float x[SEG];
#pragma unroll
      for (int j = 0; j < SEG; ++j) x[j] = nx[u][j];
#pragma unroll
      for (int kh = 0; kh < KH; ++kh) {   // feeds output row r - kh through tap row kh
        const int slot = (u - kh + KH) % KH;
#pragma unroll
        for (int c = 0; c < CO; ++c)
#pragma unroll
          for (int kw = 0; kw < KW; ++kw)
#pragma unroll
            for (int j = 0; j < 4; ++j)
              acc[slot][c][j] = kh == 0 && kw == 0 ? x[j] * w[c][0] : fmaf(x[j + kw], w[c][kh * KW + kw], acc[slot][c][j]);
      }
      load(r + U, nx[u]);
      if (r < KH - 1) continue;
      // row r - (KH - 1) is complete: its last tap row was this input row
      const int slot = (u + 1) % KH;
#pragma unroll
      for (int c = 0; c < CO; ++c) {
        if (c >= ncog) break;
        finish_row<PLAIN>(p, dst + c * p.sOc, -(at + c * sOc4) & 3, full, wo, bias[c], acc[slot][c]);
      }
      dst += p.sOh;
      at += sOh4;
    }
  }
}

// Up to four output channels per thread keep the accumulators and taps in
// registers; four with a 5 x 5 filter leave too few warps to hide the loads, so
// they go in pairs.  Two rows per thread instead of four while four would give
// fewer than six CTAs per SM, and for 1 x 1 filters, which have no halo rows to
// share; then pairs of channels for 3 x 3 too.  Measured, us, a kernel of four
// channels and four rows with loads and stores settled one by one / this: 16 x 3
// x 1280 x 1280 -> 3, 3 x 3: 320 / 219; 8 x 3 x 640 x 640 -> 3, 5 x 5: 83 / 57;
// 16 x 3 x 700 x 800 -> 4, 5 x 5: 218 / 162 (206 with four channels together); 1 x
// 3 x 1000 x 1000 -> 3, 3 x 3: 12.3 / 8.7 (14.0 with four rows); 8 x 3 x 1000 x 1000
// -> 4, 1 x 1: 62 / 42 (63 with four rows).  Six or eight rows: 268 to 275 us on the
// first.
template <int KH, int KW, int CO, int ROWS>
nk_status launch_rows_co(const Direct& p, cudaStream_t st) {
  const int cols = (p.OW + 511) / 512;
  dim3 grid((unsigned)cols * (unsigned)((p.OH + ROWS - 1) / ROWS), (unsigned)(p.N * ((p.CO + CO - 1) / CO)));
  if (p.beta == 0.f && !p.relu) (void)nk::launch_k(direct_rows_kernel<KH, KW, CO, ROWS, true>, grid, dim3(128), 0, st, 1, p, cols);
  else (void)nk::launch_k(direct_rows_kernel<KH, KW, CO, ROWS, false>, grid, dim3(128), 0, st, 1, p, cols);
  return check_launch("direct_rows_kernel");
}

template <int KH, int KW, int ROWS>
nk_status launch_rows_r(const Direct& p, int co, cudaStream_t st) {
  switch (co) {
    case 1: return launch_rows_co<KH, KW, 1, ROWS>(p, st);
    case 2: return launch_rows_co<KH, KW, 2, ROWS>(p, st);
    case 3: return launch_rows_co<KH, KW, 3, ROWS>(p, st);
    default: return launch_rows_co<KH, KW, 4, ROWS>(p, st);
  }
}

template <int KH, int KW>
nk_status launch_rows(const Direct& p, int sms, cudaStream_t st) {
  int co = p.CO < 4 ? p.CO : 4;
  const int64_t blocks = (int64_t)((p.OW + 511) / 512) * ((p.OH + 3) / 4) * p.N;
  const bool few = blocks * ((p.CO + 3) / 4) < (int64_t)sms * 6;
  if (co == 4 && (KH == 5 || (KH == 3 && few)) && (int64_t)p.N * ((p.CO + 1) / 2) <= 65535) co = 2;
  if constexpr (KH > 1)
    if (!few) return launch_rows_r<KH, KW, 4>(p, co, st);
  return launch_rows_r<KH, KW, 2>(p, co, st);
}

// `rpt` output rows per thread.
template <int KH, int KW, int CO>
nk_status launch_stream_co(const Direct& p, int rpt, cudaStream_t st) {
  dim3 grid((unsigned)((p.OW + 511) / 512), (unsigned)((p.OH + rpt - 1) / rpt), (unsigned)(p.N * ((p.CO + CO - 1) / CO)));
  if (p.beta == 0.f && !p.relu) (void)nk::launch_k(direct_stream_kernel<KH, KW, CO, true>, grid, dim3(128), 0, st, 1, p, rpt);
  else (void)nk::launch_k(direct_stream_kernel<KH, KW, CO, false>, grid, dim3(128), 0, st, 1, p, rpt);
  return check_launch("direct_stream_kernel");
}

// Stride 1, dilation 1, no program.  One input channel streams rows, except for
// 5 x 5 filters (their five accumulator rows and taps fill the registers: 16 x
// 1000 x 1000 1 -> 4, 198 us streaming, 108 by blocks of rows), 1 x 1 filters
// with several outputs (16 x 1000 x 1001 1 -> 4: 66 / 56; 1 -> 1: 22 / 25), and
// where a stream of four rows would give fewer than six CTAs per SM (2 x 300 x
// 300 1 -> 4, 3 x 3: 6.5 / 3.2).  Streams are short enough that the grid walks
// the images nearly in order, long enough to amortise the KH - 1 halo rows; us
// for 4 / 8 / 16 rows of 16 x 1000 x 1002 1 -> 4, 3 x 3: 64 / 56 / 58.
template <int KH, int KW>
nk_status launch_registers(const Direct& p, cudaStream_t st) {
  int sms = 152;
  nk_status s = require_device(&sms);
  if (s != NK_OK) return s;
  const int groups = (p.CO + 3) / 4;
  if ((int64_t)p.N * groups > 65535) return fail(NK_ERR_UNSUPPORTED, "batch x channel groups too large");
  // the limit of a grid of row blocks, which the kernels for one input channel
  // (64 rows a block at most) and for several (4) are held to
  if ((p.OH - 1) / (p.CI == 1 ? 64 : 4) >= 65535) return fail(NK_ERR_UNSUPPORTED, "output too tall");
  if constexpr (KH < 5) {
    if (p.CI == 1 && (KH == 3 || p.CO == 1)) {
      const int64_t ctas_per_row = (int64_t)((p.OW + 511) / 512) * p.N * groups;
      constexpr int64_t kRows = KH == 1 ? 4 : 8;
      int64_t rpt = (int64_t)p.OH * ctas_per_row / ((int64_t)sms * 6);
      if (rpt >= 4) {
        rpt = rpt > kRows ? kRows : rpt;
        if ((p.OH + rpt - 1) / rpt > 65535) rpt = 64;   // grid.y
        if constexpr (KH == 1) return launch_stream_co<KH, KW, 1>(p, (int)rpt, st);
        else switch (p.CO) {
          case 1: return launch_stream_co<KH, KW, 1>(p, (int)rpt, st);
          case 2: return launch_stream_co<KH, KW, 2>(p, (int)rpt, st);
          case 3: return launch_stream_co<KH, KW, 3>(p, (int)rpt, st);
          default: return launch_stream_co<KH, KW, 4>(p, (int)rpt, st);
        }
      }
    }
  }
  return launch_rows<KH, KW>(p, sms, st);
}

}  // namespace
}  // namespace nk

using namespace nk;

extern "C" nk_status nk_conv2d_nchw_fchw(const nk_tensor* I, const nk_tensor* K, nk_tensor* O,
                                         const int64_t stride[2], const int64_t dilation[2],
                                         const int64_t pad[4], const nk_epilogue* epi, void* stream) {
  nk::NvtxRange nvtx_range_("nk_conv2d_nchw_fchw");
  nk_status s = NK_OK;
  if (!I || !K || !O || !stride || !dilation || !pad) return fail(NK_ERR_INVALID_ARG, "null argument");
  if (I->rank != 4 || K->rank != 4 || O->rank != 4) return fail(NK_ERR_INVALID_ARG, "I, K, O must have rank 4");
  if (I->dtype != NK_F32 || K->dtype != NK_F32 || O->dtype != NK_F32)
    return fail(NK_ERR_UNSUPPORTED, "the direct NCHW convolution is FP32");
  if (I->stride[3] != 1 || O->stride[3] != 1) return fail(NK_ERR_UNSUPPORTED, "width must have unit stride");
  const int64_t taps = K->shape[2] * K->shape[3];
  if (K->stride[3] != 1 || K->stride[2] != K->shape[3] || K->stride[1] != taps ||
      K->stride[0] != K->shape[1] * taps)
    return fail(NK_ERR_UNSUPPORTED, "the kernel must be contiguous FCHW");
  if (I->shape[1] != K->shape[1]) return fail(NK_ERR_INVALID_ARG, "input channels differ from the kernel's");
  for (int i = 0; i < 2; ++i)
    if (stride[i] < 1 || dilation[i] < 1) return fail(NK_ERR_INVALID_ARG, "stride and dilation must be >= 1");
  for (int i = 0; i < 4; ++i)
    if (pad[i] < 0) return fail(NK_ERR_INVALID_ARG, "padding must be >= 0");
  Direct p{};
  p.N = (int)I->shape[0]; p.CI = (int)I->shape[1]; p.H = (int)I->shape[2]; p.W = (int)I->shape[3];
  p.CO = (int)K->shape[0]; p.KH = (int)K->shape[2]; p.KW = (int)K->shape[3];
  p.sh = (int)stride[0]; p.sw = (int)stride[1]; p.dh = (int)dilation[0]; p.dw = (int)dilation[1];
  p.pt = (int)pad[0]; p.pl = (int)pad[2];
  const int64_t oh = (p.H + pad[0] + pad[1] - p.dh * (p.KH - 1) - 1) / p.sh + 1;
  const int64_t ow = (p.W + pad[2] + pad[3] - p.dw * (p.KW - 1) - 1) / p.sw + 1;
  if (oh < 1 || ow < 1) return fail(NK_ERR_INVALID_ARG, "empty output");
  if (O->shape[0] != p.N || O->shape[1] != p.CO || O->shape[2] != oh || O->shape[3] != ow)
    return fail(NK_ERR_INVALID_ARG, "O must be [%d,%d,%lld,%lld]", p.N, p.CO, (long long)oh, (long long)ow);
  p.OH = (int)oh; p.OW = (int)ow;
  if (taps > 64) return fail(NK_ERR_UNSUPPORTED, "more than 64 filter taps");
  p.in_h = (TH - 1) * p.sh + (p.KH - 1) * p.dh + 1;
  p.in_w = (TW - 1) * p.sw + (p.KW - 1) * p.dw + 1;
  if (p.in_h > MAX_IN_H || p.in_w > MAX_IN_W)
    return fail(NK_ERR_UNSUPPORTED, "stride/dilation/filter too large for the direct kernel's halo tile");
  p.I = static_cast<const float*>(I->ptr);
  p.sIn = I->stride[0]; p.sIc = I->stride[1]; p.sIh = I->stride[2];
  p.Kr = static_cast<const float*>(K->ptr);
  p.O = static_cast<float*>(O->ptr);
  p.sOn = O->stride[0]; p.sOc = O->stride[1]; p.sOh = O->stride[2];
  const nk_epilogue e0{nullptr, 0, 0, 1.f, 1.f, nullptr, nullptr, nullptr};
  const nk_epilogue& E = epi ? *epi : e0;
  p.bias = E.bias;
  p.relu = E.relu;
  p.beta = E.accumulate ? 1.f : 0.f;
  if (E.pro_a || E.pro_b)
    return fail(NK_ERR_UNSUPPORTED, "the direct NCHW convolution takes no operand prologue");
  if ((s = ew_program(E.ew, O, &p.ew, "ew")) != NK_OK) return s;
  if ((s = require_device()) != NK_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // The register-streaming kernels carry no epilogue program (a call in
  // their loops would slow the plain path); a program goes to the general
  // kernel below.
  const bool plain = p.ew.n == 0;
  if (plain && p.sh == 1 && p.sw == 1 && p.dh == 1 && p.dw == 1) {
    if (p.KH == 3 && p.KW == 3) return launch_registers<3, 3>(p, st);
    if (p.KH == 5 && p.KW == 5) return launch_registers<5, 5>(p, st);
    if (p.KH == 1 && p.KW == 1) return launch_registers<1, 1>(p, st);
  }
  const int groups = (p.CO + CO_G - 1) / CO_G;
  if ((int64_t)p.N * groups > 65535) return fail(NK_ERR_UNSUPPORTED, "batch x channel groups too large");
  dim3 grid((unsigned)((p.OW + TW - 1) / TW), (unsigned)((p.OH + TH - 1) / TH), (unsigned)(p.N * groups));
  if (grid.y > 65535) return fail(NK_ERR_UNSUPPORTED, "output too tall");
  const size_t smem = (size_t)(CO_G * 64 + p.in_h * p.in_w) * sizeof(float);
  (void)nk::launch_k(direct_conv_kernel, dim3(grid), dim3(THREADS), smem, st, 1, p);
  return check_launch("direct_conv_kernel");
}
