// tc_gemm.cuh -- linalg.matmul on the 5th-generation tensor cores: the kernel,
// its parameters and its launch (shared by k_tc_gemm.cu and k_tc_gemm_ew.cu).
//
// C[m,n] (+)= sum_k A[m,k] B[k,n] (Sec. 2.1.1 Listing "linalg-matmul") with
// the bias / ReLU epilogue of the lowered Linear layer (Sec. 2.1.2 Listing
// "listing1").  The paper tiles the loop nest and searches tile sizes
// (Sec. 4.3); here one tile is a 128 x BN block of C computed by one CTA of a
// persistent grid:
//
//   warp 0      TMA producer: A and B tiles (128-byte rows, 128B swizzle) into
//               a STAGES-deep shared-memory ring, one mbarrier pair per slot.
//               Every CTA loads its own tiles: a cluster of two is a CTA pair
//               (below), in which each CTA loads its half of B; no TMA load
//               is multicast.
//   warp 1      allocates TMEM; one thread issues tcgen05.mma (M=128, N=BN,
//               K=16 BF16 / K=32 E4M3 per instruction) into a double-buffered
//               FP32 accumulator in TMEM, and tcgen05.commit frees each slot.
//   warps 2..5  epilogue: tcgen05.ld of their 32-lane quarter, then
//               alpha, beta*C, bias, ReLU and stores -- overlapping the
//               next tile's main loop through the second accumulator.
//
// BF16x3 sums hi*hi, hi*lo and lo*hi per K step: on one CTA in two MMAs, hi *
// [hi lo] over two adjacent accumulators and lo * hi into the second.  Split-K
// writes each slice's raw tile to the workspace and a fixed-order reduce pass
// applies the epilogue.
//
// Every wait is bounded (see tc_ptx.cuh); on a timeout the CTA drains its own
// copies and MMAs, frees TMEM and exits, and the host reports NK_ERR_TIMEOUT.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include "nk_internal.cuh"
#include "tc_ptx.cuh"

namespace nk {

// Output tile of the convolution: NB images x R output rows x Q output
// columns (NB*R*Q <= 128 GEMM rows), and the input walk for each filter tap.
struct ConvTile {
  int Q, R, NB;
  int tiles_w, tiles_h;
  int N, OH, OW;
  int sh, sw, dh, dw, pt, pl;
  int KW, cblocks;
  int cblk;               // channels per K block: one 128-byte row (64 BF16, 128 E4M3)
};

struct TcParams {
  CUtensorMap tmA, tmB, tmA2, tmB2;
  int M, N, K;
  int bn, stages;
  int tiles_m, tiles_n;   // tiles_m padded to the cluster size
  int splits, kb_per_split, nkb;
  int units;
  float* C;
  int64_t ldc;
  float* partial;         // [splits][M][ldp] when splits > 1
  int ldp;                // row stride of a partial tile: N rounded up to 4 floats
  int part_vec;           // partial is 16-byte aligned
  const float* bias;
  int bias_on_m, relu;
  float beta, alpha;
  const float* scale_a;
  const float* scale_b;
  int64_t budget;
  int c_vec;
  // grouped launches: per-group shapes, outputs and TMA descriptors in device memory
  const struct GroupDesc* groups;
  const int* tile_start;        // [G+1] prefix sums of tiles per group
  const int* unit_group;        // [units] group of each unit, or null (binary search)
  const CUtensorMap* gmaps;     // [G][2]: A_g, Bt_g
  const CUtensorMap* gcmaps;    // [G]: C_g for the TMA-store epilogue (c_tma), or null
  int G;
  // implicit-GEMM convolution (tmA: 4-D NHWC input map, tmB: 3-D [F][taps][C] map)
  ConvTile cv;
  uint32_t a_box_bytes;         // bytes TMA writes per A stage (16 KB unless a conv tile is short)
  // epilogue through shared memory and TMA stores (plain GEMM, beta = 0, one K slice)
  CUtensorMap tmC;
  int c_tma;                    // 1: TMA stores; 2: C has no tensor map, the warp copies the box out
  int boxes2;                   // c_tma: two staging boxes per epilogue warp
  EwProg ew;                    // fused elementwise program (offsets from C), single launches
  int out_bf16;                 // single convolutions: C holds BF16 (RNE of the FP32 result)
  int c_vec32;                  // single convolutions: 32-byte aligned output rows
  int resid;                    // single convolutions: ew is {ADD t, RELU}, t with 32-byte aligned rows
};

struct GroupDesc {
  int M, N, K, tiles_n;
  float* C;
  int64_t ldc;
  float beta;
  int kblocks;            // K blocks of 64 elements (a conv: taps x channel blocks)
  const float* bias;      // per output column, or null
  int relu;
  int pad;
  ConvTile cv;            // grouped convolutions: the group's output tiling
};

// Launches the variant that runs p's elementwise program in registers before
// the TMA-store epilogue (k_tc_gemm_ew.cu), and its failure word.
nk_status tc_gemm_ew_launch(const TcParams& p, const nk_schedule& s, int kind, bool ep8, int grid, int smem,
                            cudaStream_t st);
uint32_t tc_ew_read_and_clear_errors();

namespace {

__device__ unsigned int g_tc_err;   // one per translation unit (see kErrTimeout)

inline uint32_t read_and_clear_err() {
  unsigned int v = 0;
  if (cudaMemcpyFromSymbol(&v, g_tc_err, sizeof v) != cudaSuccess) return 0;
  const unsigned int z = 0;
  cudaMemcpyToSymbol(g_tc_err, &z, sizeof z);
  return v;
}

constexpr int kThreads = 192;       // 6 warps
constexpr int kBM = 128;
constexpr int kRowBytes = 128;      // one K block = one 128-byte swizzle row
constexpr int kGroupM = 8;          // rasterisation: 8 (pair-)rows of tiles per band
constexpr int kMaxSmem = 232448;    // 227 KB opt-in limit

// Epilogue staging: one 32 x 32 FP32 box (4 KB, 128B-swizzled) per epilogue warp.
constexpr int kStageBox = 4096;
__host__ __device__ inline int staging_bytes(bool wide, int mch = 1) {
  return mch > 1 ? 0 : (wide ? 8 : 4) * kStageBox;   // tall tiles store directly
}

// One pipeline stage: mch A tiles of 128 rows (one per accumulator chain)
// and one B^T tile of bn rows, each row 128 bytes; BF16x3 doubles it (hi, lo).
__host__ __device__ inline int stage_bytes(int kind, int bn, int mch = 1) {
  const int ab = mch * kBM * kRowBytes + bn * kRowBytes;
  return kind == TC_BF16X3 ? 2 * ab : ab;
}

struct Unit {
  int tm, tn, split;
};

// Everything one role needs to know about a unit of work.
struct UnitView {
  int tm, tn, split, kb0, kb1, M, N;
  const CUtensorMap* ma;
  const CUtensorMap* mb;
  const CUtensorMap* mc;   // C map of the TMA-store epilogue
  float* C;
  int64_t ldc;
  float beta;
  const float* bias;
  int relu;
  const ConvTile* cv;    // conv launches: the tiling of this unit's convolution
};

__device__ __forceinline__ Unit decode_unit(const TcParams& p, int u, int cl, int rank) {
  const int tmp_count = p.tiles_m / cl;
  const int per_split = tmp_count * p.tiles_n;
  Unit r;
  r.split = u / per_split;
  const int t = u % per_split;
  const int band = kGroupM * p.tiles_n;
  const int first = (t / band) * kGroupM;
  const int gm = min(tmp_count - first, kGroupM);
  const int tmp = first + (t % band) % gm;
  r.tn = (t % band) / gm;
  r.tm = tmp * cl + rank;
  return r;
}

template <bool GROUPED>
__device__ __forceinline__ UnitView view_unit(const TcParams& p, int u, int cl, int rank) {
  UnitView v;
  if constexpr (GROUPED) {
    // group g with tile_start[g] <= u < tile_start[g+1]: one load from a
    // plan's unit map, else a binary search of the prefix sums.  The map
    // took 0.270 -> 0.245 ms off 512 uneven groups: the search's dependent
    // loads ran in every role for every unit.
    int lo = 0;
    if (p.unit_group) {
      lo = __ldg(p.unit_group + u);
    } else {
      int hi = p.G;
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(p.tile_start + mid) <= u) lo = mid;
        else hi = mid;
      }
    }
    const GroupDesc& g = p.groups[lo];
    const int t = u - __ldg(p.tile_start + lo);
    v.tm = (t / g.tiles_n) * cl + rank;   // a pair's tile: its two 128-row halves
    v.tn = t % g.tiles_n;
    v.split = 0;
    v.kb0 = 0;
    v.kb1 = g.kblocks;
    v.M = g.M;
    v.N = g.N;
    v.ma = p.gmaps + 2 * lo;
    v.mb = p.gmaps + 2 * lo + 1;
    v.mc = p.gcmaps ? p.gcmaps + lo : nullptr;
    v.C = g.C;
    v.ldc = g.ldc;
    v.beta = g.beta;
    v.bias = g.bias;
    v.relu = g.relu;
    v.cv = &g.cv;
  } else {
    const Unit t = decode_unit(p, u, cl, rank);
    v.tm = t.tm;
    v.tn = t.tn;
    v.split = t.split;
    v.kb0 = t.split * p.kb_per_split;
    v.kb1 = min(p.nkb, v.kb0 + p.kb_per_split);
    v.M = p.M;
    v.N = p.N;
    v.ma = &p.tmA;
    v.mb = &p.tmB;
    v.mc = &p.tmC;
    v.C = p.C;
    v.ldc = p.ldc;
    v.beta = p.beta;
    v.bias = p.bias;
    v.relu = p.relu;
    v.cv = &p.cv;
  }
  return v;
}

// Output row of GEMM row r (0..127) of conv tile tm, or -1 if it is padding.
__device__ __forceinline__ int conv_row(const ConvTile& c, int tm, int r) {
  if (r >= c.Q * c.R * c.NB) return -1;
  const int tw = tm % c.tiles_w;
  const int th = (tm / c.tiles_w) % c.tiles_h;
  const int tb = tm / (c.tiles_w * c.tiles_h);
  const int q = r % c.Q, rr = (r / c.Q) % c.R, b = r / (c.Q * c.R);
  const int n = tb * c.NB + b, oh = th * c.R + rr, ow = tw * c.Q + q;
  if (n >= c.N || oh >= c.OH || ow >= c.OW) return -1;
  return (n * c.OH + oh) * c.OW + ow;
}

// PAIR: the two CTAs of a cluster form one 2-SM MMA (cta_group::2) computing a
// 256 x BN tile; each holds its 128 rows of A and BN/2 rows of B^T, and the
// even CTA's barriers gate the pair (its MMA thread is the only issuer).
//
// WIDE: a pair computing a 256 x 512 tile as two independent N = 256
// accumulator chains that share the A tile.  One chain of dependent MMAs on a
// single accumulator issues about one instruction per ~190 cycles, while an
// N = 256 MMA holds only 128 cycles of math; interleaving two chains hides
// that latency.  Both chains fill the 512 TMEM columns, so the accumulator is
// single-buffered and eight epilogue warps drain it.
//
// For BF16x3 a wide tile is 256 x 256: its two N = 256 accumulators are hi*hi
// and the corrections.
//
// MCH > 1 (tall tile, one CTA): MCH stacked 128-row tiles of A share one B
// tile, each with its own accumulator chain, so narrow problems (N = 64, 128)
// keep several independent MMA chains in flight.
//
// EP8 (GEMMs with one CTA per SM, single and grouped): eight epilogue warps,
// two per TMEM lane quarter, each draining half of a tile's columns -- the
// epilogue of a 128 x 256 tile would otherwise outlast the next tile's MMAs.
// Each warp has its own staging boxes for the TMA-store epilogue.
//
// Grouped launches store through TMA too (c_tma with a C map per group,
// when every group overwrites a 16-byte aligned C whose rows end on 16-byte
// boundaries): the store clips each group's ragged rows and columns past the
// last 16-byte granule, and one instruction writes a 32 x 32 block where
// per-lane stores touch 32 rows.  On 512 uneven groups (128 x 256 tiles,
// 4 stages) 0.244 -> 0.234 ms.
//
// EW: single GEMMs whose elementwise program runs in registers before the
// TMA-store epilogue.  A variant of its own, because the inlined operations
// would cost every plain epilogue registers; without it a program goes
// through a local buffer and row-per-lane stores.  Bias + GELU on 4096 x 4096 x
// 1024 (BF16 operands): 354 us with an interpreter call per element and scalar
// stores, 133 us with this epilogue's earlier form, 46.6 us now.
template <int KIND, int CL, bool GROUPED, bool CONV = false, bool PAIR = false, bool WIDE = false, int MCH = 1,
          bool EP8 = false, bool EW = false>
__global__ void __launch_bounds__((WIDE || EP8) ? 320 : 192, (WIDE || EP8 || KIND == TC_BF16X3) ? 1 : 2) tc_gemm_kernel(const __grid_constant__ TcParams p) {
  static_assert(!EP8 || (!WIDE && MCH == 1 && !CONV), "eight epilogue warps: plain GEMM tiles");
  static_assert(PAIR == (CL == 2), "a cluster of two is a CTA pair, and a CTA pair is a cluster of two");
  static_assert(!WIDE || (PAIR && !GROUPED), "wide tiles are pair tiles");
  static_assert(MCH == 1 || (!PAIR && !GROUPED && KIND != TC_BF16X3 && CL == 1), "tall tiles: one CTA");
  static_assert(!EW || (!GROUPED && !CONV && MCH == 1), "programs in registers: single GEMMs with TMA stores");
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = ptx::smem_u32(smem_raw);
  const uint32_t base = (raw + 1023) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - raw);

  const int b_rows_smem = PAIR ? p.bn / 2 : p.bn;   // rows of B^T this CTA keeps per stage
  const int sb = stage_bytes(KIND, b_rows_smem, MCH);
  const int S = p.stages;
  const uint32_t stg0 = base + S * sb;   // epilogue staging boxes
  const int stg_bytes = staging_bytes(WIDE || EP8, MCH) << p.boxes2;
  const uint32_t bar0 = stg0 + stg_bytes;   // full[S], empty[S], tfull[2], tempty[2], drain
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (S + s); };
  auto tfull_bar = [&](int b) { return bar0 + 8u * (2 * S + b); };
  auto tempty_bar = [&](int b) { return bar0 + 8u * (2 * S + 2 + b); };
  const uint32_t drain_bar = bar0 + 8u * (2 * S + 4);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base_ptr + S * sb + stg_bytes + 8 * (2 * S + 5));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  {
    // Guard: the launch must have given this layout enough dynamic shared
    // memory; otherwise report and leave before touching any of it.
    uint32_t dsz;
    asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dsz));
    const uint32_t need = (base - raw) + (uint32_t)(S * sb + stg_bytes + 8 * (2 * S + 5) + 8);
    if (need > dsz) {
      if (threadIdx.x == 0) atomicOr(&g_tc_err, 2u);
      return;
    }
  }

  const int warp = threadIdx.x / 32;
  const int lane = threadIdx.x % 32;
  const int rank = CL == 2 ? (int)ptx::cluster_ctarank() : 0;
  const int cluster_id = blockIdx.x / CL;
  const int n_clusters = gridDim.x / CL;
  // Accumulator columns per buffer: BN, or 2*BN for BF16x3 (hi*hi and the
  // hi*lo + lo*hi corrections accumulate apart and meet in the epilogue, so
  // the large term sees K/16 roundings instead of 3K/16).
  const int acc_cols = KIND == TC_BF16X3 ? 2 * p.bn : MCH * p.bn;
  const uint32_t tmem_cols = WIDE ? 512u : 2u * (uint32_t)acc_cols < 32u ? 32u : 2u * (uint32_t)acc_cols;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      ptx::mbar_init(full_bar(s), 1);
      ptx::mbar_init(empty_bar(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(tfull_bar(b), 1);
      ptx::mbar_init(tempty_bar(b), (WIDE || (PAIR && EP8)) ? 16 : (PAIR || EP8) ? 8 : 4);   // every epilogue warp
    }
    ptx::mbar_init(drain_bar, 1);
    *abort_flag = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 0 && lane == 0 && !GROUPED) {
    ptx::tma_prefetch_desc(&p.tmA);
    ptx::tma_prefetch_desc(&p.tmB);
    if (KIND == TC_BF16X3) {
      ptx::tma_prefetch_desc(&p.tmA2);
      ptx::tma_prefetch_desc(&p.tmB2);
    }
  }
  if (warp == 1) {
    if (PAIR) {
      ptx::tmem_alloc_pair(ptx::smem_u32(tmem_slot), tmem_cols);
      ptx::tmem_relinquish_pair();
    } else {
      ptx::tmem_alloc(ptx::smem_u32(tmem_slot), tmem_cols);
      ptx::tmem_relinquish();
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  if (CL == 2) ptx::cluster_sync();
  const uint32_t tmem_base = *tmem_slot;
  // Set-up above touched no global data; everything below runs after the
  // earlier kernels on the stream have finished.
  nk::pdl_wait();
  nk::pdl_trigger();

  const int a_bytes = MCH * kBM * kRowBytes;
  const int b_bytes = b_rows_smem * kRowBytes;
  // Stage layout: [A][B] or, for BF16x3, [A_hi][A_lo][B_hi][B_lo] on one CTA
  // (B_hi and B_lo adjacent: one B operand of 2 * bn rows), and
  // [A_hi][B_hi][A_lo][B_lo] on a pair.
  constexpr bool HILO = KIND == TC_BF16X3 && !PAIR;
  auto a_smem = [&](int s, int part) { return base + s * sb + part * (HILO ? a_bytes : a_bytes + b_bytes); };
  auto b_smem = [&](int s, int part) {
    return base + s * sb + (HILO ? 2 * a_bytes + part * b_bytes : part * (a_bytes + b_bytes) + a_bytes);
  };

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      int it = 0;
      const int kblk = KIND == TC_FP8 ? 128 : 64;   // elements per 128-byte row
      bool ok = true;
      for (int u = cluster_id; u < p.units && ok; u += n_clusters) {
        const UnitView t = view_unit<GROUPED>(p, u, CL, rank);
        const int kb0 = t.kb0;
        const int kb1 = t.kb1;
        for (int kb = kb0; kb < kb1; ++kb, ++it) {
          const int s = it % S;
          const uint32_t ph = (uint32_t)(it / S) & 1u;
          if (!ptx::mbar_wait(empty_bar(s), ph ^ 1u, p.budget, abort_flag, &g_tc_err)) { ok = false; break; }
          if constexpr (PAIR) {
            // Both CTAs load their own halves; the even CTA's barrier counts both.
            const uint32_t lf = ptx::mapa(full_bar(s), 0);
            const int by = t.tn * p.bn + rank * b_rows_smem;
            if constexpr (CONV) {
              const ConvTile& c = *t.cv;
              if (rank == 0) ptx::mbar_arrive_expect_tx(full_bar(s), 2u * (p.a_box_bytes + (uint32_t)b_bytes));
              const int tap = kb / c.cblocks, c0 = (kb % c.cblocks) * c.cblk;
              const int kh = tap / c.KW, kw = tap % c.KW;
              const int tw = t.tm % c.tiles_w, th = (t.tm / c.tiles_w) % c.tiles_h;
              const int tb = t.tm / (c.tiles_w * c.tiles_h);
              ptx::tma_load_4d_pair(a_smem(s, 0), t.ma, lf, c0, tw * c.Q * c.sw + kw * c.dw - c.pl,
                                    th * c.R * c.sh + kh * c.dh - c.pt, tb * c.NB);
              ptx::tma_load_3d_pair(b_smem(s, 0), t.mb, lf, c0, tap, by);
            } else {
              if (rank == 0) ptx::mbar_arrive_expect_tx(full_bar(s), 2u * (uint32_t)sb);
              const int kx = kb * kblk;
              if (WIDE && KIND != TC_BF16X3) {
                // chain h (N columns h*256 .. h*256+255): this CTA holds its 128 rows of B^T
                ptx::tma_load_2d_pair(a_smem(s, 0), t.ma, lf, kx, t.tm * kBM);
                ptx::tma_load_2d_pair(b_smem(s, 0), t.mb, lf, kx, t.tn * p.bn + rank * 128);
                ptx::tma_load_2d_pair(b_smem(s, 0) + 128 * kRowBytes, t.mb, lf, kx, t.tn * p.bn + 256 + rank * 128);
                continue;
              }
              const int nparts = KIND == TC_BF16X3 ? 2 : 1;
              for (int part = 0; part < nparts; ++part) {
                ptx::tma_load_2d_pair(a_smem(s, part), part ? &p.tmA2 : t.ma, lf, kx, t.tm * kBM);
                ptx::tma_load_2d_pair(b_smem(s, part), part ? &p.tmB2 : t.mb, lf, kx, by);
              }
            }
            continue;
          }
          if constexpr (CONV) {
            // K block kb = (filter tap, 64-channel block); the A box is the
            // input window that tap sees, shifted and strided by TMA.
            const ConvTile& c = *t.cv;
            // bytes one A box writes (a short conv tile writes fewer than 16 KB)
            const uint32_t a_box = GROUPED ? (uint32_t)(c.Q * c.R * c.NB * kRowBytes) : p.a_box_bytes;
            ptx::mbar_arrive_expect_tx(full_bar(s), MCH * a_box + (uint32_t)b_bytes);
            const int tap = kb / c.cblocks, c0 = (kb % c.cblocks) * c.cblk;
            const int kh = tap / c.KW, kw = tap % c.KW;
            for (int ch = 0; ch < MCH; ++ch) {
              const int ct = t.tm * MCH + ch;   // conv tile of this chain
              const int tw = ct % c.tiles_w, th = (ct / c.tiles_w) % c.tiles_h;
              const int tb = ct / (c.tiles_w * c.tiles_h);
              ptx::tma_load_4d(a_smem(s, 0) + ch * kBM * kRowBytes, t.ma, full_bar(s), c0,
                               tw * c.Q * c.sw + kw * c.dw - c.pl, th * c.R * c.sh + kh * c.dh - c.pt, tb * c.NB);
            }
            ptx::tma_load_3d(b_smem(s, 0), t.mb, full_bar(s), c0, tap, t.tn * p.bn);
            continue;
          }
          ptx::mbar_arrive_expect_tx(full_bar(s), (uint32_t)sb);
          const int kx = kb * kblk;
          const int ay = t.tm * MCH * kBM;
          const int by = t.tn * p.bn;
          const int nparts = KIND == TC_BF16X3 ? 2 : 1;
          for (int part = 0; part < nparts; ++part) {
            const CUtensorMap* ma = part ? &p.tmA2 : t.ma;
            const CUtensorMap* mb = part ? &p.tmB2 : t.mb;
            for (int ch = 0; ch < MCH; ++ch)
              ptx::tma_load_2d(a_smem(s, part) + ch * kBM * kRowBytes, ma, full_bar(s), kx, ay + ch * kBM);
            ptx::tma_load_2d(b_smem(s, part), mb, full_bar(s), kx, by);
          }
        }
      }
      // Drain: the last copy issued into each slot must land before exit.  In
      // a pair the odd CTA cannot poll the even CTA's barrier; the MMA that
      // consumed its copies frees its own slot, so it waits on that instead.
      const int last = it;
      for (int j = last - 1; j >= 0 && j >= last - S; --j) {
        if (PAIR && rank != 0) ptx::mbar_drain(empty_bar(j % S), (uint32_t)(j / S) & 1u, 100000000ull);
        else ptx::mbar_drain(full_bar(j % S), (uint32_t)(j / S) & 1u, 100000000ull);
      }
    }
  } else if (warp == 1) {
    // -------------------------------------------------------------- MMA
    if (lane == 0 && (!PAIR || rank == 0)) {
      const uint32_t idesc = ptx::make_idesc(KIND == TC_FP8 ? 0 : 1, PAIR ? 2 * kBM : kBM, WIDE ? 256 : p.bn);
      const uint32_t idesc2 = HILO ? ptx::make_idesc(1, kBM, 2 * p.bn) : 0u;
      int it = 0, tc = 0;
      bool ok = true;
      for (int u = cluster_id; u < p.units && ok; u += n_clusters, ++tc) {
        const UnitView t = view_unit<GROUPED>(p, u, CL, rank);
        const int kb0 = t.kb0;
        const int kb1 = t.kb1;
        const int acc = WIDE ? 0 : tc & 1;   // a wide tile's two chains fill TMEM: one buffer
        const uint32_t aph = WIDE ? (uint32_t)tc & 1u : (uint32_t)(tc >> 1) & 1u;
        if (!ptx::mbar_wait(tempty_bar(acc), aph ^ 1u, p.budget, abort_flag, &g_tc_err)) break;
        ptx::tc_fence_after();
        const uint32_t d = tmem_base + (uint32_t)(acc * acc_cols);
        const uint32_t d2 = d + (uint32_t)(WIDE ? 256 : p.bn);   // BF16x3 corrections / second wide chain
        for (int kb = kb0; kb < kb1; ++kb, ++it) {
          const int s = it % S;
          const uint32_t ph = (uint32_t)(it / S) & 1u;
          if (!ptx::mbar_wait(full_bar(s), ph, p.budget, abort_flag, &g_tc_err)) { ok = false; break; }
          ptx::tc_fence_after();
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const uint32_t koff = (uint32_t)k * 32u;
            const uint64_t ad = ptx::sw128_desc(a_smem(s, 0) + koff);
            const uint64_t bd = ptx::sw128_desc(b_smem(s, 0) + koff);
            const uint32_t accum = (kb > kb0 || k > 0) ? 1u : 0u;
            if constexpr (HILO) {
              // hi * [hi lo] in one MMA over both accumulators, then lo * hi.
              // An MMA of this kernel takes about as long at N = 128 as at
              // 256, so two a step instead of three: 4096^3, with its casts,
              // 364 -> 329 us (L2 now bounds it: see x3_wide_wins).
              ptx::tc_mma<0>(d, ad, bd, idesc2, accum);
              ptx::tc_mma<0>(d2, ptx::sw128_desc(a_smem(s, 1) + koff), bd, idesc, 1u);
              continue;
            }
            if (PAIR) ptx::tc_mma_pair<KIND == TC_FP8>(d, ad, bd, idesc, accum);
            else ptx::tc_mma<KIND == TC_FP8>(d, ad, bd, idesc, accum);
#pragma unroll
            for (int ch = 1; ch < MCH; ++ch)   // further chains: their own A rows, the same B
              ptx::tc_mma<KIND == TC_FP8>(d + (uint32_t)(ch * p.bn),
                                          ptx::sw128_desc(a_smem(s, 0) + ch * kBM * kRowBytes + koff), bd, idesc,
                                          accum);
            if (WIDE && KIND != TC_BF16X3) {   // second chain: B^T rows 128..255 of this CTA's stage
              const uint64_t bw = ptx::sw128_desc(b_smem(s, 0) + 128 * kRowBytes + koff);
              ptx::tc_mma_pair<KIND == TC_FP8>(d2, ad, bw, idesc, accum);
            }
            if constexpr (KIND == TC_BF16X3 && PAIR) {
              const uint64_t ad2 = ptx::sw128_desc(a_smem(s, 1) + koff);
              const uint64_t bd2 = ptx::sw128_desc(b_smem(s, 1) + koff);
              ptx::tc_mma_pair<0>(d2, ad, bd2, idesc, accum);   // hi * lo
              ptx::tc_mma_pair<0>(d2, ad2, bd, idesc, 1u);      // lo * hi
            }
          }
          if (PAIR) ptx::tc_commit_pair_mc(empty_bar(s), (uint16_t)0x3);
          else ptx::tc_commit(empty_bar(s));
        }
        if (!ok) break;
        if (PAIR) ptx::tc_commit_pair_mc(tfull_bar(acc), (uint16_t)0x3);
        else ptx::tc_commit(tfull_bar(acc));
      }
      // Drain: every MMA this thread issued completes before TMEM is freed.
      if (PAIR) ptx::tc_commit_pair(drain_bar);
      else ptx::tc_commit(drain_bar);
      ptx::mbar_drain(drain_bar, 0, 100000000ull);
    }
  } else {
    // ---------------------------------------------------------- epilogue
    const int q = warp & 3;   // TMEM lane quarter this warp may read
    float alpha = p.alpha;
    if (p.scale_a) alpha = __frcp_rn(__fmul_rn(*p.scale_a, *p.scale_b));
    int tc = 0;
    uint32_t nst = 0;   // stores this warp has staged
    for (int u = cluster_id; u < p.units; u += n_clusters, ++tc) {
      const UnitView t = view_unit<GROUPED>(p, u, CL, rank);
      const int acc = WIDE ? 0 : tc & 1;
      const uint32_t aph = WIDE ? (uint32_t)tc & 1u : (uint32_t)(tc >> 1) & 1u;
      if (!ptx::mbar_wait(tfull_bar(acc), aph, p.budget, abort_flag, &g_tc_err)) break;
      ptx::tc_fence_after();
      auto release = [&] {   // this warp has read its part of the accumulator
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (PAIR) ptx::mbar_arrive_cluster(ptx::mapa(tempty_bar(acc), 0));   // the issuer's barrier
          else ptx::mbar_arrive(tempty_bar(acc));
        }
      };
      if constexpr (!CONV && MCH == 1) {
        if (p.c_tma) {
          // Coalesced epilogue: registers -> this warp's 128B-swizzled 32 x 32
          // staging box -> one TMA store (rows / columns past C are clipped).
          // What bounds it is latency -- TMEM load, staging, the wait until
          // the box's previous store has read it -- with one or two warps per
          // scheduler, so two segments' TMEM loads share one wait, a warp
          // alternates between two boxes where shared memory has room for
          // them, and the accumulator goes back to the MMA warp after its last
          // load, not after its last store.
          // Alone, on one GB300: 4096 x 4096 x 1024 BF16 47.1 -> 35.6 us on wide
          // pair tiles and 39.0 -> 35.1 us on 128 x 256 tiles (eight warps); with
          // a bias, whose columns used to be 32 predicated scalar loads, 66.4 ->
          // 37.0 and 89.4 -> 35.5 us; 8192^3 609 -> 560 us; FP8 4096^3 79 -> 53 us.
          const int row = t.tm * kBM + q * 32 + lane;
          const bool row_ok = row < t.M;
          const int c_cols = (WIDE || EP8) ? p.bn / 2 : p.bn;   // eight warps: two per lane quarter, half the columns each
          const int c_begin = (WIDE || EP8) ? ((warp - 2) / 4) * c_cols : 0;
          const int col_begin = t.tn * p.bn + c_begin;
          const int nseg = max(0, min(c_cols, t.N - col_begin) + 31) / 32;
          const uint32_t ta0 = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * acc_cols + c_begin);
          const float bm = (t.bias && p.bias_on_m && row_ok) ? t.bias[row] : 0.f;
          constexpr int PARTS = KIND == TC_BF16X3 ? 2 : 1;
          // segments whose TMEM loads share one wait (a program's steps need the
          // registers of the second: bias + GELU on 4096 x 4096 x 1024 44.5 us with
          // two, 43.8 with one)
          constexpr int AHEAD = EW ? 1 : 2 / PARTS;
          auto load = [&](int i, uint32_t (&r)[PARTS][32]) {
            ptx::tmem_ld32_async(ta0 + 32u * i, r[0]);
            if constexpr (PARTS == 2) ptx::tmem_ld32_async(ta0 + 32u * i + (uint32_t)p.bn, r[1]);
          };
          auto emit = [&](int i, const uint32_t (&r)[PARTS][32]) {
            const int col0 = col_begin + 32 * i;
            float v[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) {
              v[j] = __uint_as_float(r[0][j]);
              if constexpr (PARTS == 2) v[j] += __uint_as_float(r[1][j]);
              v[j] *= alpha;
            }
            if (t.bias) {
              if (p.bias_on_m) {
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] += bm;
              } else if (col0 + 32 <= t.N && (reinterpret_cast<uintptr_t>(t.bias + col0) & 15) == 0) {
#pragma unroll
                for (int j = 0; j < 32; j += 4) {
                  const float4 b = *reinterpret_cast<const float4*>(t.bias + col0 + j);
                  v[j] += b.x; v[j + 1] += b.y; v[j + 2] += b.z; v[j + 3] += b.w;
                }
              } else {
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] += col0 + j < t.N ? t.bias[col0 + j] : 0.f;
              }
            }
            if (t.relu) {
#pragma unroll
              for (int j = 0; j < 32; ++j) v[j] = (v[j] > 0.f || v[j] != v[j]) ? v[j] : 0.f;
            }
            // the program reads its operands (which may alias C) before the
            // segment is staged, and so before any of it is stored
            if constexpr (EW)
              ew_regs(p.ew, v, row_ok ? (t.N - col0 < 32 ? t.N - col0 : 32) : 0, (int64_t)row * t.ldc + col0);
            const uint32_t stg = stg0 + (uint32_t)((((warp - 2) << p.boxes2) + (int)(nst & (uint32_t)p.boxes2)) * kStageBox);
            ++nst;
            if (lane == 0) {   // the box's previous store has read it
              if (p.boxes2) ptx::bulk_wait_read1();
              else ptx::bulk_wait_read0();
            }
            __syncwarp();
#pragma unroll
            for (int j16 = 0; j16 < 8; ++j16) {
              const uint32_t addr = stg + (uint32_t)(lane * 128 + ((j16 ^ (lane & 7)) * 16));
              asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v[4 * j16]), "f"(v[4 * j16 + 1]),
                           "f"(v[4 * j16 + 2]), "f"(v[4 * j16 + 3])
                           : "memory");
            }
            if (p.c_tma == 2) {
              // rows of C that no TMA store can address (N or the row stride
              // not a multiple of 4, or a C off 16 bytes): the warp writes the
              // box row by row, 128 contiguous bytes each, where a lane per
              // row touched 32 sectors with every store: BF16x3 3001
              // x 2002 x 1999, whole call, 104 -> 87 us.
              __syncwarp();
              const int rows = min(32, t.M - (t.tm * kBM + q * 32));
              float* dst = t.C + (int64_t)(t.tm * kBM + q * 32) * t.ldc + col0 + lane;
              const bool in = col0 + lane < t.N;
#pragma unroll 8
              for (int r = 0; r < rows; ++r) {
                float x;
                asm volatile("ld.shared.f32 %0, [%1];"
                             : "=f"(x)
                             : "r"(stg + (uint32_t)(r * 128 + (((lane >> 2) ^ (r & 7)) * 16) + (lane & 3) * 4))
                             : "memory");
                if (in) dst[(int64_t)r * t.ldc] = x;
              }
              __syncwarp();
              return;
            }
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
              ptx::tma_store_2d(t.mc, stg, col0, t.tm * kBM + q * 32);
              ptx::bulk_commit();
            }
          };
          if (nseg == 0) release();
#pragma unroll 1
          for (int i = 0; i < nseg; i += AHEAD) {
            uint32_t r[AHEAD][PARTS][32];
#pragma unroll
            for (int h = 0; h < AHEAD; ++h)
              if (i + h < nseg) load(i + h, r[h]);
            ptx::tmem_wait_ld(r[0][0]);
#pragma unroll
            for (int h = 0; h < AHEAD * PARTS; ++h)
              if (h > 0) ptx::tmem_after_wait(r[h / PARTS][h % PARTS]);
            if (i + AHEAD >= nseg) release();
#pragma unroll
            for (int h = 0; h < AHEAD; ++h)
              if (i + h < nseg) emit(i + h, r[h]);
          }
          continue;
        }
      }
      for (int ch = 0; ch < MCH; ++ch) {   // chains of a tall tile (one otherwise)
      const int tmc = t.tm * MCH + ch;
      const int row = CONV ? conv_row(*t.cv, tmc, q * 32 + lane) : tmc * kBM + q * 32 + lane;
      const bool row_ok = CONV ? row >= 0 : row < t.M;
      // a wide tile has two warps per lane quarter, each draining one chain's 256 columns
      const int c_begin = (WIDE || EP8) ? ((warp - 2) / 4) * (p.bn / 2) : 0;
      const int c_end = (WIDE || EP8) ? c_begin + p.bn / 2 : p.bn;
      for (int c0 = c_begin; c0 < c_end; c0 += 32) {
        float v[32];
        const uint32_t ta =
            tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * acc_cols + ch * p.bn + c0);
        ptx::tmem_ld32(ta, v);
        if (KIND == TC_BF16X3) {
          float w[32];
          ptx::tmem_ld32(ta + (uint32_t)p.bn, w);
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] += w[j];
        }
        const int col0 = t.tn * p.bn + c0;
        if (!row_ok || col0 >= t.N) continue;
        if (p.partial) {
          float* dst = p.partial + ((int64_t)t.split * p.M + row) * p.ldp + col0;
          if (p.part_vec && col0 + 32 <= p.ldp) {
#pragma unroll
            for (int j = 0; j < 32; j += 4)
              *reinterpret_cast<float4*>(dst + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j)
              if (col0 + j < p.N) dst[j] = v[j];
          }
          continue;
        }
        if constexpr (CONV && !GROUPED) {
          if (p.c_vec32 && t.beta == 0.f && col0 + 32 <= t.N && (p.ew.n == 0 || p.resid)) {
            // Full 32-column segment, no accumulate, and no program or the
            // residual program ADD t, RELU (inline, the interpreter's FP32
            // steps): one code path for FP32 and BF16 outputs.
            const int64_t off = (int64_t)row * t.ldc + col0;
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] *= alpha;
            if (t.bias) add_bias32(t.bias + col0, v);
            if (t.relu) {
#pragma unroll
              for (int j = 0; j < 32; ++j) v[j] = (v[j] > 0.f || v[j] != v[j]) ? v[j] : 0.f;
            }
            if (p.resid) {
              const float4* tr = reinterpret_cast<const float4*>(p.ew.t[0] + off);
#pragma unroll
              for (int j = 0; j < 32; j += 4) {
                const float4 r4 = tr[j / 4];
                const float rv[4] = {r4.x, r4.y, r4.z, r4.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                  const float x = __fadd_rn(v[j + e], rv[e]);
                  v[j + e] = (x > 0.f || x != x) ? x : 0.f;
                }
              }
            }
            if (p.out_bf16) store32_bf16_v8(reinterpret_cast<__nv_bfloat16*>(t.C) + off, v);
            else store32_f32_v8(t.C + off, v);
            continue;
          }
          if (p.out_bf16) {
            // BF16 output: the FP32 epilogue, then one RNE rounding per value
            __nv_bfloat16* dh = reinterpret_cast<__nv_bfloat16*>(t.C) + (int64_t)row * t.ldc + col0;
            const int ncol = t.N - col0 < 32 ? t.N - col0 : 32;
            __align__(16) float buf[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) {
              float x = alpha * v[j];
              if (j < ncol) {
                if (t.beta != 0.f) x = fmaf(t.beta, __bfloat162float(dh[j]), x);
                if (t.bias) x += t.bias[col0 + j];
                if (t.relu) x = (x > 0.f || x != x) ? x : 0.f;
              }
              buf[j] = x;
            }
            if (p.ew.n) ew_apply(p.ew, buf, ncol, (int64_t)row * t.ldc + col0);
            if (p.c_vec && ncol == 32) {
              store32_bf16(dh, buf);
            } else {
              for (int j = 0; j < ncol; ++j) dh[j] = __float2bfloat16_rn(buf[j]);
            }
            continue;
          }
        }
        float* dst = t.C + (int64_t)row * t.ldc + col0;
        const float bm = (t.bias && p.bias_on_m) ? t.bias[row] : 0.f;
        const float beta = t.beta;
        if (!CONV && p.c_vec32 && beta == 0.f && col0 + 32 <= t.N && p.ew.n == 0) {
          // full 32-column segment of 32-byte aligned rows: 32-byte stores
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            float x = alpha * v[j];
            if (t.bias) x += p.bias_on_m ? bm : t.bias[col0 + j];
            if (t.relu) x = (x > 0.f || x != x) ? x : 0.f;
            v[j] = x;
          }
          store32_f32_v8(dst, v);
          continue;
        }
        if (p.ew.n) {
          // A program runs out of line.  The segment goes through a local
          // buffer: the program reads its operands (which may alias C) before
          // the store, and v[] is not live across the call, so the plain
          // paths below keep their registers.
          const int ncol = t.N - col0 < 32 ? t.N - col0 : 32;
          __align__(16) float buf[32];
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            float x = alpha * v[j];
            if (j < ncol) {
              if (beta != 0.f) x = fmaf(beta, dst[j], x);
              if (t.bias) x += p.bias_on_m ? bm : t.bias[col0 + j];
              if (t.relu) x = (x > 0.f || x != x) ? x : 0.f;
            }
            buf[j] = x;
          }
          ew_apply(p.ew, buf, ncol, (int64_t)row * t.ldc + col0);
          if (p.c_vec32 && ncol == 32) store32_f32_v8(dst, buf);
          else
            for (int j = 0; j < ncol; ++j) dst[j] = buf[j];
        } else if (p.c_vec && col0 + 32 <= t.N) {
          // the segment of C_in in flight at once, before the first store
          float4 cin[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            cin[j] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (beta != 0.f) cin[j] = *reinterpret_cast<const float4*>(dst + 4 * j);
          }
#pragma unroll
          for (int j = 0; j < 32; j += 4) {
            float o[4];
            const float ci[4] = {cin[j / 4].x, cin[j / 4].y, cin[j / 4].z, cin[j / 4].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              float x = alpha * v[j + e];
              if (beta != 0.f) x = fmaf(beta, ci[e], x);
              if (t.bias) x += p.bias_on_m ? bm : t.bias[col0 + j + e];
              if (t.relu) x = (x > 0.f || x != x) ? x : 0.f;
              o[e] = x;
            }
            *reinterpret_cast<float4*>(dst + j) = make_float4(o[0], o[1], o[2], o[3]);
          }
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            if (col0 + j >= t.N) continue;
            float x = alpha * v[j];
            if (beta != 0.f) x = fmaf(beta, dst[j], x);
            if (t.bias) x += p.bias_on_m ? bm : t.bias[col0 + j];
            if (t.relu) x = (x > 0.f || x != x) ? x : 0.f;
            dst[j] = x;
          }
        }
      }
      }
      release();
    }
    if (!CONV && p.c_tma && lane == 0) ptx::bulk_wait0();   // every store has landed
  }

  ptx::tc_fence_before();
  __syncthreads();
  // A pair frees TMEM only once the even CTA has drained every MMA that
  // writes into either CTA's TMEM.
  if (CL == 2) ptx::cluster_sync();
  ptx::tc_fence_after();
  if (warp == 1) {
    if (PAIR) ptx::tmem_dealloc_pair(tmem_base, tmem_cols);
    else ptx::tmem_dealloc(tmem_base, tmem_cols);
  }
  if (CL == 2) ptx::cluster_sync();
}

template <int KIND, int CL, bool GROUPED = false, bool CONV = false, bool PAIR = false, bool WIDE = false,
          int MCH = 1, bool EP8 = false, bool EW = false>
nk_status launch(const TcParams& p, int grid, int smem, cudaStream_t st) {
  auto kern = tc_gemm_kernel<KIND, CL, GROUPED, CONV, PAIR, WIDE, MCH, EP8, EW>;
  // the attribute is set once per device and size (it stays set on the function)
  static int set_bytes[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || set_bytes[dev] < smem) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(tc_gemm_kernel)");
    if (dev >= 0 && dev < 64) set_bytes[dev] = smem;
  }
  const cudaError_t e = nk::launch_k(kern, dim3(grid), dim3((WIDE || EP8) ? 320 : kThreads), smem, st, CL, p);
  if (e != cudaSuccess) return cuda_fail(e, "launch tc_gemm_kernel");
  return check_launch("tc_gemm_kernel");
}

// The kernel of a single GEMM's schedule.  EP8: eight epilogue warps.  EW: with
// its program in registers (BF16 and FP8; tall tiles, mch > 1, have no
// TMA-store epilogue and so no such variant).
template <bool EW, bool EP8>
nk_status launch_single(const TcParams& p, const nk_schedule& s, int kind, int mch, int grid, int smem,
                        cudaStream_t st) {
  if constexpr (!EP8 && !EW) {
    if (kind == TC_BF16X3 && s.tile_n == 256)
      return launch<TC_BF16X3, 2, false, false, true, true>(p, grid, smem, st);
  }
  if constexpr (!EP8) {
    if (s.tile_n == 512) {
      if (kind == TC_FP8) return launch<TC_FP8, 2, false, false, true, true, 1, false, EW>(p, grid, smem, st);
      return launch<TC_BF16, 2, false, false, true, true, 1, false, EW>(p, grid, smem, st);
    }
    if constexpr (!EW) {
      if (mch == 2) {
        if (kind == TC_FP8) return launch<TC_FP8, 1, false, false, false, false, 2>(p, grid, smem, st);
        return launch<TC_BF16, 1, false, false, false, false, 2>(p, grid, smem, st);
      }
      if (mch == 4) {
        if (kind == TC_FP8) return launch<TC_FP8, 1, false, false, false, false, 4>(p, grid, smem, st);
        return launch<TC_BF16, 1, false, false, false, false, 4>(p, grid, smem, st);
      }
    }
  }
  const bool pair = s.tile_m == 256;
  if constexpr (!EW) {
    if (kind == TC_BF16X3)
      return pair ? launch<TC_BF16X3, 2, false, false, true, false, 1, EP8>(p, grid, smem, st)
                  : launch<TC_BF16X3, 1, false, false, false, false, 1, EP8>(p, grid, smem, st);
  }
  if (kind == TC_FP8)
    return pair ? launch<TC_FP8, 2, false, false, true, false, 1, EP8, EW>(p, grid, smem, st)
                : launch<TC_FP8, 1, false, false, false, false, 1, EP8, EW>(p, grid, smem, st);
  return pair ? launch<TC_BF16, 2, false, false, true, false, 1, EP8, EW>(p, grid, smem, st)
              : launch<TC_BF16, 1, false, false, false, false, 1, EP8, EW>(p, grid, smem, st);
}

}  // namespace
}  // namespace nk
