// k_tc_gemm.cu -- host side of the tcgen05 GEMM (tc_gemm.cuh): tensor maps,
// schedules, split-K, the per-tap implicit-GEMM convolution and the grouped
// plans.  Programs in registers are launched from k_tc_gemm_ew.cu, compiled
// beside this file.
#include <cuda.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <climits>
#include <cstring>
#include <mutex>
#include <vector>

#include "tc_gemm.cuh"

namespace nk {

uint32_t tc_read_and_clear_errors() { return read_and_clear_err() | tc_ew_read_and_clear_errors(); }

namespace {

// ------------------------------------------------------------------ host
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// 2-D K-major operand [rows, K] with row stride ld (elements), 128B swizzle.
nk_status make_kmajor_map(CUtensorMap* m, bool fp8, const void* ptr, int64_t rows, int64_t K,
                          int64_t ld, int box_rows) {
  auto fn = encode_fn();
  if (!fn) return fail(NK_ERR_CUDA, "cuTensorMapEncodeTiled is unavailable");
  const int esz = fp8 ? 1 : 2;
  cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)(ld * esz)};
  cuuint32_t box[2] = {(cuuint32_t)(kRowBytes / esz), (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  CUresult r = fn(m, fp8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                  const_cast<void*>(ptr), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS)
    return fail(NK_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d) for a [%lld, %lld] operand", (int)r,
                (long long)rows, (long long)K);
  return NK_OK;
}

int smem_bytes(int kind, int bn, int stages, bool wide = false, int mch = 1) {
  return 1024 + stages * stage_bytes(kind, bn, mch) + staging_bytes(wide, mch) + 8 * (2 * stages + 5) + 16;
}

// Accumulator chains along M of a one-CTA schedule: tile_m 256 / 512 with
// cluster 1 are tall tiles of 2 / 4 chains (tile_m 256 with cluster 2 is a pair).
int chains_of(const nk_schedule& s) { return (s.cluster == 1 && s.tile_m > 128) ? s.tile_m / 128 : 1; }

// Wide tiles: 512 columns, or 256 of BF16x3 (two accumulators), fill the TMEM.
bool is_wide(int kind, const nk_schedule& s) { return s.tile_n == 512 || (kind == TC_BF16X3 && s.tile_n == 256); }

// BF16x3 with no schedule given: 256 x 256 tiles on CTA pairs where they win.
// A 128 x 128 tile loads 64 KB for 768 cycles of MMAs, more than L2 delivers;
// a CTA of the wide pair loads 64 KB for 1536, but its accumulators have no
// second buffer, so every tile's epilogue is exposed.  Microseconds of a wave,
// fitted: 0.62 per 64-deep K block + 1.5 (128 x 128), 1.0 + 6 (wide).  Whole
// calls, 128 x 128 against wide: 4096^3 329 / 311 us, 4096 x 4096 x 1024 92 /
// 96, 1024 x 4096 x 1024 33.0 / 32.2, 3001 x 2002 x 1999 87 / 99.  The schedule
// space, whose points the stored corpora time one by one, does not hold this one:
// it cannot be asked for, and a caller's schedule is always taken as it is.
bool x3_wide_wins(int M, int N, int K, int sms) {
  const int64_t wide = (int64_t)((M + 255) / 256) * ((N + 255) / 256);
  const int64_t square = (int64_t)((M + 127) / 128) * ((N + 127) / 128);
  const int64_t pairs = sms / 2;
  const double nkb = (K + 63) / 64;
  return (wide + pairs - 1) / pairs * (1.0 * nkb + 6.0) < (square + sms - 1) / sms * (0.62 * nkb + 1.5);
}

// Shared memory of a schedule: a CTA of a pair (tile_m 256) keeps half of B.
int smem_of(int kind, const nk_schedule& s) {
  const bool pair = s.cluster == 2 && s.tile_m == 256;
  return smem_bytes(kind, pair ? s.tile_n / 2 : s.tile_n, s.stages, is_wide(kind, s), chains_of(s));
}

// CTAs that fit on one SM: shared memory and the 512 TMEM columns.
int ctas_per_sm(int kind, const nk_schedule& s) {
  if (is_wide(kind, s)) return 1;   // a wide tile holds all 512 TMEM columns
  const int bn = s.tile_n;
  const int sm = smem_of(kind, s);
  int by_smem = kMaxSmem / sm;
  const int acc = kind == TC_BF16X3 ? 2 * bn : chains_of(s) * bn;
  int cols = 2 * acc < 32 ? 32 : 2 * acc;
  int by_tmem = 512 / cols;
  int r = by_smem < by_tmem ? by_smem : by_tmem;
  return r < 1 ? 1 : (r > 2 ? 2 : r);
}

}  // namespace

bool tc_schedule_valid(int kind, const nk_schedule& s, int M, int N, int K) {
  (void)M; (void)N; (void)K;
  // tile_m 256 with cluster 2 = a CTA pair issuing 2-SM MMAs; tile_m 256 / 512
  // with cluster 1 = a tall tile of 2 / 4 accumulator chains sharing B.  A
  // cluster of two is always a CTA pair: no schedule multicasts a TMA load.
  if (s.tile_m != 128 && s.tile_m != 256 && s.tile_m != 512) return false;
  if (s.cluster == 2 && s.tile_m != 256) return false;
  if (chains_of(s) > 1 && (kind == TC_BF16X3 || chains_of(s) * s.tile_n > 256)) return false;
  if (s.tile_n != 64 && s.tile_n != 128 && s.tile_n != 256 && s.tile_n != 512) return false;
  if (s.tile_n == 512 && (s.tile_m != 256 || kind == TC_BF16X3)) return false;   // wide pair tiles only
  if (kind == TC_BF16X3 && s.tile_n > 128) return false;   // 2 accumulators x 2 buffers <= 512 cols
  if (s.tile_k != (kind == TC_FP8 ? 128 : 64)) return false;
  if (s.cluster != 1 && s.cluster != 2) return false;
  if (s.split_k < 1 || s.split_k > 32) return false;
  if (s.stages < 2 || s.stages > 8) return false;
  if (smem_of(kind, s) > kMaxSmem) return false;
  return true;
}

nk_schedule tc_default_schedule(int kind, int M, int N, int K, int sms) {
  nk_schedule s{};
  s.tile_m = 128;
  s.tile_k = kind == TC_FP8 ? 128 : 64;
  s.tile_n = kind == TC_BF16X3 ? 128 : 256;
  if (N <= 64) s.tile_n = 64;
  else if (N <= 128) s.tile_n = 128;
  s.cluster = 1;
  s.stages = 2;
  while (s.stages < 8 && smem_bytes(kind, s.tile_n, s.stages + 1) <= kMaxSmem) ++s.stages;
  // Large BF16 / FP8 problems: wide pair tiles (256 x 512, two MMA chains)
  // when there are at least two waves of them.
  if (kind != TC_BF16X3 && (int64_t)((M + 255) / 256) * ((N + 511) / 512) >= sms) {
    s.tile_m = 256; s.tile_n = 512; s.cluster = 2; s.stages = 4; s.split_k = 1;
    return s;
  }
  // Split K when the output tiles cannot fill the GPU and K is deep.
  const int tiles = ((M + 127) / 128) * ((N + s.tile_n - 1) / s.tile_n);
  const int nkb = (K + s.tile_k - 1) / s.tile_k;
  s.split_k = 1;
  while (tiles * s.split_k * 2 <= sms && nkb / (s.split_k * 2) >= 4 && s.split_k < 16) s.split_k *= 2;
  return s;
}

// Split-K partials: rows of N rounded up to 16 bytes, so that every row takes
// 16-byte stores and loads.
static int partial_ld(int N) { return (N + 3) / 4 * 4; }

size_t tc_gemm_ws(const TcGemm& g, const nk_schedule& s) {
  if (s.split_k <= 1) return 0;
  return (size_t)s.split_k * g.M * partial_ld(g.N) * sizeof(float);
}

nk_status tc_gemm(const TcGemm& g, const nk_schedule& sched, void* ws, size_t ws_bytes, cudaStream_t st) {
  nk_schedule s = sched;
  int sms = 0;
  nk_status status = require_device(&sms);
  if (status != NK_OK) return status;
  if (g.M <= 0 || g.N <= 0) return NK_OK;
  if (!tc_schedule_valid(g.kind, s, g.M, g.N, g.K))
    return fail(NK_ERR_NO_SCHEDULE, "illegal tensor-core schedule");
  if (g.any_schedule && g.kind == TC_BF16X3 && s.split_k == 1 && x3_wide_wins(g.M, g.N, g.K, sms))
    s = nk_schedule{256, 256, 64, 2, 3, 1};
  if (g.K <= 0) {
    // Empty reduction: the epilogue alone (the CUDA-core kernel with K = 0).
    SimtGemm z{};
    z.A = nullptr; z.sam = 0; z.sak = 1;
    z.B = nullptr; z.sbk = 1; z.sbn = 0;
    z.C = g.C; z.scm = g.ldc; z.scn = 1;
    z.bias = g.bias; z.bias_on_m = g.bias_on_m;
    z.M = g.M; z.N = g.N; z.K = 0;
    z.alpha = 1.f; z.beta = g.beta; z.relu = g.relu;
    z.ew = g.ew;
    return simt_gemm(z, 64, 1, nullptr, 0, st);
  }
  const bool fp8 = g.kind == TC_FP8;
  const int esz = fp8 ? 1 : 2;
  if ((g.lda * esz) % 16 || (g.ldb * esz) % 16)
    return fail(NK_ERR_MISALIGNED, "operand row strides must be multiples of 16 bytes");
  TcParams p;
  memset(&p, 0, sizeof p);
  const int CL = s.cluster;
  if ((status = make_kmajor_map(&p.tmA, fp8, g.A, g.M, g.K, g.lda, kBM)) != NK_OK) return status;
  const int b_box = s.tile_n == 512 ? 128 : s.tile_n / CL;   // a wide tile loads B^T in 128-row boxes
  if ((status = make_kmajor_map(&p.tmB, fp8, g.B, g.N, g.K, g.ldb, b_box)) != NK_OK) return status;
  if (g.kind == TC_BF16X3) {
    if ((status = make_kmajor_map(&p.tmA2, fp8, g.A2, g.M, g.K, g.lda, kBM)) != NK_OK) return status;
    if ((status = make_kmajor_map(&p.tmB2, fp8, g.B2, g.N, g.K, g.ldb, s.tile_n / CL)) != NK_OK) return status;
  }
  p.M = g.M; p.N = g.N; p.K = g.K;
  p.bn = s.tile_n;
  p.stages = s.stages;
  const int mch = chains_of(s);
  const int tm = (g.M + kBM * mch - 1) / (kBM * mch);
  p.tiles_m = (tm + CL - 1) / CL * CL;
  p.tiles_n = (g.N + s.tile_n - 1) / s.tile_n;
  p.nkb = (g.K + s.tile_k - 1) / s.tile_k;
  int splits = s.split_k > p.nkb ? p.nkb : s.split_k;
  p.kb_per_split = (p.nkb + splits - 1) / splits;
  splits = (p.nkb + p.kb_per_split - 1) / p.kb_per_split;
  p.splits = splits;
  p.units = (p.tiles_m / CL) * p.tiles_n * splits;
  p.C = g.C;
  p.ldc = g.ldc;
  p.partial = nullptr;
  if (splits > 1) {
    const size_t need = (size_t)splits * g.M * partial_ld(g.N) * sizeof(float);
    if (!ws || ws_bytes < need) return fail(NK_ERR_WORKSPACE, "split-K needs %zu bytes of workspace", need);
    p.partial = static_cast<float*>(ws);
    p.ldp = partial_ld(g.N);
    p.part_vec = (reinterpret_cast<uintptr_t>(ws) & 15) == 0;
  }
  p.bias = g.bias;
  p.bias_on_m = g.bias_on_m;
  p.relu = g.relu;
  p.beta = g.beta;
  p.alpha = g.alpha;
  p.scale_a = g.scale_a;
  p.scale_b = g.scale_b;
  p.ew = g.ew;
  p.budget = wait_budget();
  const bool cvec = ((reinterpret_cast<uintptr_t>(g.C) & 15) == 0) && (g.ldc % 4 == 0);
  p.c_vec = cvec ? 1 : 0;
  p.c_vec32 = (splits == 1 && (reinterpret_cast<uintptr_t>(g.C) & 31) == 0 && g.ldc % 8 == 0) ? 1 : 0;
  // Staged epilogue: plain overwrite of C in one K slice, by TMA stores where C
  // is 16-byte aligned.  Rows must also end on a 16-byte boundary (N % 4 == 0):
  // a TMA store clips the innermost dimension only to 16-byte granules, so
  // with N % 4 != 0 and a padded row stride it wrote the row's padding (caught
  // by canaries).  Any other C is copied out by the warps.
  p.c_tma = 0;
  if (mch == 1 && splits == 1 && g.beta == 0.f && (g.ew.n == 0 || g.kind != TC_BF16X3)) {
    p.c_tma = 2;
    auto fn = encode_fn();
    cuuint64_t dims[2] = {(cuuint64_t)g.N, (cuuint64_t)g.M};
    cuuint64_t strides[1] = {(cuuint64_t)(g.ldc * 4)};
    cuuint32_t box[2] = {32, 32};
    cuuint32_t es[2] = {1, 1};
    if ((reinterpret_cast<uintptr_t>(g.C) & 15) == 0 && (g.ldc * 4) % 16 == 0 && g.N % 4 == 0 && fn &&
        fn(&p.tmC, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, g.C, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
           CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS)
      p.c_tma = 1;
  }
  int smem = smem_of(g.kind, s);
  const int per_sm = ctas_per_sm(g.kind, s);
  const bool wide = is_wide(g.kind, s);
  // Eight epilogue warps when a CTA has the SM to itself, and a second staging
  // box per warp where shared memory has room beside the SM's CTAs.
  const bool ep8 = p.c_tma && !wide && per_sm == 1 && smem + 4 * kStageBox <= kMaxSmem;
  if (ep8) smem += 4 * kStageBox;
  p.boxes2 = p.c_tma && per_sm * (smem + staging_bytes(wide || ep8)) <= kMaxSmem ? 1 : 0;
  if (p.boxes2) smem += staging_bytes(wide || ep8);
  int grid = sms * per_sm;
  grid = grid / CL * CL;
  const int need_ctas = p.units * CL;
  if (grid > need_ctas) grid = need_ctas;
  if (grid < CL) grid = CL;
  if (p.ew.n && p.c_tma) status = tc_gemm_ew_launch(p, s, g.kind, ep8, grid, smem, st);
  else if (ep8) status = launch_single<false, true>(p, s, g.kind, mch, grid, smem, st);
  else status = launch_single<false, false>(p, s, g.kind, mch, grid, smem, st);
  if (status != NK_OK || splits == 1) return status;
  SplitReduce r{};
  r.partial = p.partial;
  r.ldp = p.ldp;
  r.splits = splits;
  r.M = g.M;
  r.N = g.N;
  r.C = g.C;
  r.scm = g.ldc;
  r.scn = 1;
  r.bias = g.bias;
  r.bias_on_m = g.bias_on_m;
  r.alpha = g.alpha;
  r.beta = g.beta;
  r.relu = g.relu;
  r.scale_a = g.scale_a;
  r.scale_b = g.scale_b;
  r.ew = g.ew;
  return splitk_reduce(r, st);
}

}  // namespace nk

// ===================================================================== conv
namespace nk {
namespace {

// Output tile (Q columns x R rows x NB images, <= 128 GEMM rows) with the
// fewest tiles; ties go to the widest rows.
ConvTile search_conv_tile(const ConvGeom& g, int maxrows) {
  ConvTile best{};
  int64_t best_tiles = INT64_MAX;
  for (int Q = 1; Q <= maxrows && Q <= g.ow; ++Q) {
    if (Q * g.sw > 256) break;
    for (int R = 1; Q * R <= maxrows && R <= g.oh; ++R) {
      if (R * g.sh > 256) break;
      const int NB = std::max(1, std::min(g.n, maxrows / (Q * R)));
      const int64_t tiles = (int64_t)((g.n + NB - 1) / NB) * ((g.oh + R - 1) / R) * ((g.ow + Q - 1) / Q);
      if (tiles < best_tiles || (tiles == best_tiles && Q > best.Q)) {
        best_tiles = tiles;
        best.Q = Q; best.R = R; best.NB = NB;
      }
    }
  }
  best.tiles_w = (g.ow + best.Q - 1) / best.Q;
  best.tiles_h = (g.oh + best.R - 1) / best.R;
  best.N = g.n; best.OH = g.oh; best.OW = g.ow;
  best.sh = g.sh; best.sw = g.sw; best.dh = g.dh; best.dw = g.dw; best.pt = g.pt; best.pl = g.pl;
  best.KW = g.kw;
  best.cblk = 64;
  best.cblocks = (g.c + 63) / 64;
  return best;
}

// The search above runs per call; its answer is cached per geometry.
std::mutex g_ctile_mu;
std::vector<std::pair<ConvGeom, ConvTile>> g_ctile_cache;

ConvTile cached_conv_tile(const ConvGeom& g) {
  std::lock_guard<std::mutex> lk(g_ctile_mu);
  for (auto& e : g_ctile_cache)
    if (std::memcmp(&e.first, &g, sizeof g) == 0) return e.second;
  const ConvTile t = search_conv_tile(g, 128);
  if (g_ctile_cache.size() > 4096) g_ctile_cache.clear();
  g_ctile_cache.push_back({g, t});
  return t;
}

// The tile of a geometry, with K blocks of one 128-byte row of channels.
ConvTile choose_conv_tile(const ConvGeom& g, int kind) {
  ConvTile t = cached_conv_tile(g);
  t.cblk = kind == TC_FP8 ? 128 : 64;
  t.cblocks = (g.c + t.cblk - 1) / t.cblk;
  return t;
}

nk_status make_conv_maps(CUtensorMap* map_a, CUtensorMap* map_b, const TcConv& c, const ConvTile& t, int bn_box) {
  auto fn = encode_fn();
  if (!fn) return fail(NK_ERR_CUDA, "cuTensorMapEncodeTiled is unavailable");
  const ConvGeom& g = c.g;
  const bool fp8 = c.kind == TC_FP8;
  const int esz = fp8 ? 1 : 2;
  const CUtensorMapDataType dt = fp8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  {
    cuuint64_t dims[4] = {(cuuint64_t)g.c, (cuuint64_t)g.w, (cuuint64_t)g.h, (cuuint64_t)g.n};
    cuuint64_t strides[3] = {(cuuint64_t)c.sI_w * esz, (cuuint64_t)c.sI_h * esz, (cuuint64_t)c.sI_n * esz};
    cuuint32_t box[4] = {(cuuint32_t)t.cblk, (cuuint32_t)(t.Q * g.sw), (cuuint32_t)(t.R * g.sh), (cuuint32_t)t.NB};
    cuuint32_t es[4] = {1, (cuuint32_t)g.sw, (cuuint32_t)g.sh, 1};
    CUresult r = fn(map_a, dt, 4, const_cast<void*>(c.I), dims, strides, box,
                    es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(NK_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d) for the conv input", (int)r);
  }
  {
    const int taps = g.kh * g.kw;
    cuuint64_t dims[3] = {(cuuint64_t)g.c, (cuuint64_t)taps, (cuuint64_t)c.F};
    cuuint64_t strides[2] = {(cuuint64_t)c.ldw * esz, (cuuint64_t)c.sW_f * esz};
    cuuint32_t box[3] = {(cuuint32_t)t.cblk, 1, (cuuint32_t)bn_box};
    cuuint32_t es[3] = {1, 1, 1};
    CUresult r = fn(map_b, dt, 3, const_cast<void*>(c.Wt), dims, strides, box,
                    es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(NK_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d) for the conv weights", (int)r);
  }
  return NK_OK;
}

}  // namespace

bool tc_conv_schedule_valid(const ConvGeom& g, int F, const nk_schedule& s, int kind) {
  if (kind != TC_BF16 && kind != TC_FP8) return false;
  if (halo_schedule(g, s, kind)) return halo_schedule_valid(g, F, s, kind);
  if (g.sw > 8 || g.sh > 8 || s.tile_n == 512) return false;
  // E4M3 convolutions: one CTA per tile, tall tiles included (no CTA pairs)
  if (kind == TC_FP8 && s.cluster == 2) return false;
  return tc_schedule_valid(kind, s, g.n * g.oh * g.ow, F, g.kh * g.kw * g.c);
}

// The shared-window kernel where it wins (see tc_halo_default_schedule).
// Otherwise one 128 x 64 tile per CTA for BF16 (128 x 128 for E4M3 when F >
// 64) -- more, narrower tiles keep more independent MMA chains busy: over the
// tuner's BF16 corpus (100 conv problems, every legal schedule timed) 64-wide
// tiles took the mean regret of this default from 16 % to 6 %, mostly on
// strided and 1x1 layers with F >= 128 -- with as many stages as leave room
// for two CTAs per SM (short K loops gain more from a second CTA than from
// deeper rings), and split-K while the grid would leave half the SMs idle.
nk_schedule tc_conv_default_schedule(const ConvGeom& g, int F, int sms, int kind) {
  bool ok = false;
  if (kind == TC_BF16 || kind == TC_FP8) {
    nk_schedule h = tc_halo_default_schedule(g, F, sms, &ok, kind);
    if (ok) return h;
  }
  nk_schedule s{};
  s.tile_m = 128;
  s.tile_k = kind == TC_FP8 ? 128 : 64;
  s.tile_n = (kind == TC_BF16 || F <= 64) ? 64 : 128;
  s.cluster = 1;
  s.split_k = 1;
  s.stages = 2;
  const bool two = 4 * s.tile_n <= 512;   // two CTAs' double-buffered accumulators fit in TMEM
  for (;;) {
    nk_schedule n = s;
    n.stages = s.stages + 1;
    const int need = smem_of(kind, n);
    if (n.stages > 8 || need > kMaxSmem || (two && 2 * (need + 1024) > kMaxSmem + 1024)) break;
    s = n;
  }
  const ConvTile t = choose_conv_tile(g, kind);
  const int ctiles = t.tiles_w * t.tiles_h * ((g.n + t.NB - 1) / t.NB);
  const int tiles = ctiles * ((F + s.tile_n - 1) / s.tile_n);
  const int nkb = g.kh * g.kw * t.cblocks;
  // More than a wave of two CTAs per SM, and enough K blocks to cover a tile's
  // epilogue (with fewer than 16, a wave and a half): 256 x 128 tiles on CTA
  // pairs (three stages, so that two CTAs still share an SM), which read the
  // filters half as often.  128 x 64 tiles / pairs, us: 128x56x56x64 -> 128 3x3 /
  // 2 32.4 / 22.4, 64x28x28x128 -> 256 3x3 / 2 21.3 / 15.6, 128x14x14x256 -> 512
  // 3x3 / 2 37.1 / 23.5; with one wave, 32x28x28x128 -> 256 3x3 / 2 13.0 / 14.0;
  // with four K blocks, 128x14x14x256 -> 512 1x1 / 2 8.5 / 9.0.
  if (kind == TC_BF16 && F > 64 && ((tiles > 2 * sms && nkb >= 16) || (tiles > 3 * sms && nkb >= 8)))
    return nk_schedule{256, 128, 64, 2, 3, 1};
  while (tiles * s.split_k * 2 <= sms && nkb / (s.split_k * 2) >= 4 && s.split_k < 16) s.split_k *= 2;
  return s;
}

size_t tc_conv_ws(const TcConv& c, const nk_schedule& s) {
  if (s.split_k <= 1 || halo_schedule(c.g, s, c.kind)) return 0;
  return (size_t)s.split_k * c.g.n * c.g.oh * c.g.ow * partial_ld(c.F) * sizeof(float);
}

nk_status tc_conv(const TcConv& c, const nk_schedule& s, void* ws, size_t ws_bytes, cudaStream_t st) {
  int sms = 0;
  nk_status status = require_device(&sms);
  if (status != NK_OK) return status;
  const ConvGeom& g = c.g;
  const int kind = c.kind;
  if ((kind == TC_BF16 || kind == TC_FP8) && halo_schedule(g, s, kind)) return tc_halo_conv(c, s, st);
  const int M = g.n * g.oh * g.ow;
  if (g.sw > 8 || g.sh > 8) return fail(NK_ERR_UNSUPPORTED, "conv stride above 8");
  if (!tc_conv_schedule_valid(g, c.F, s, kind))
    return fail(NK_ERR_NO_SCHEDULE, "illegal tensor-core schedule for conv");
  const int esz = kind == TC_FP8 ? 1 : 2;
  if ((c.sI_w * esz) % 16 || (c.sI_h * esz) % 16 || (c.sI_n * esz) % 16 || (c.ldw * esz) % 16 ||
      (c.sW_f * esz) % 16 || (reinterpret_cast<uintptr_t>(c.I) & 15) || (reinterpret_cast<uintptr_t>(c.Wt) & 15))
    return fail(NK_ERR_MISALIGNED, "conv operands need 16-byte aligned bases and strides");
  const ConvTile t = choose_conv_tile(g, kind);
  TcParams p;
  memset(&p, 0, sizeof p);
  const int CL = s.cluster;
  if ((status = make_conv_maps(&p.tmA, &p.tmB, c, t, s.tile_n / CL)) != NK_OK) return status;
  p.cv = t;
  p.a_box_bytes = (uint32_t)(t.Q * t.R * t.NB * kRowBytes);
  p.M = M; p.N = c.F; p.K = g.kh * g.kw * g.c;
  p.bn = s.tile_n;
  p.stages = s.stages;
  const int mch = chains_of(s);
  const int ctiles = t.tiles_w * t.tiles_h * ((g.n + t.NB - 1) / t.NB);
  const int tm = (ctiles + mch - 1) / mch;
  p.tiles_m = (tm + CL - 1) / CL * CL;
  p.tiles_n = (c.F + s.tile_n - 1) / s.tile_n;
  p.nkb = g.kh * g.kw * t.cblocks;
  int splits = s.split_k > p.nkb ? p.nkb : s.split_k;
  p.kb_per_split = (p.nkb + splits - 1) / splits;
  splits = (p.nkb + p.kb_per_split - 1) / p.kb_per_split;
  p.splits = splits;
  p.units = (p.tiles_m / CL) * p.tiles_n * splits;
  p.C = c.O;
  p.ldc = c.F;
  if (splits > 1) {
    const size_t need = (size_t)splits * M * partial_ld(c.F) * sizeof(float);
    if (!ws || ws_bytes < need) return fail(NK_ERR_WORKSPACE, "split-K needs %zu bytes of workspace", need);
    p.partial = static_cast<float*>(ws);
    p.ldp = partial_ld(c.F);
    p.part_vec = (reinterpret_cast<uintptr_t>(ws) & 15) == 0;
  }
  p.bias = c.bias;
  p.relu = c.relu;
  p.beta = c.beta;
  // E4M3 operands the caller quantised carry 1/(s_i s_w) in alpha
  p.alpha = (kind == TC_FP8 && !c.scale_i) ? c.alpha : 1.f;
  p.scale_a = c.scale_i;   // E4M3: alpha = 1 / (s_i * s_w), read on the device
  p.scale_b = c.scale_w;
  p.ew = c.ew;
  p.budget = wait_budget();
  p.out_bf16 = c.out_bf16;
  p.c_vec32 = (splits == 1 && (reinterpret_cast<uintptr_t>(c.O) & 31) == 0 && c.F % (c.out_bf16 ? 16 : 8) == 0) ? 1 : 0;
  p.resid = (c.ew.n == 2 && c.ew.op[0] == NK_EW_ADD && c.ew.op[1] == NK_EW_RELU &&
             (reinterpret_cast<uintptr_t>(c.ew.t[0]) & 31) == 0 && c.F % 8 == 0) ? 1 : 0;
  // vector stores: 16-byte aligned rows (FP32: F % 4, BF16: F % 8)
  p.c_vec = ((reinterpret_cast<uintptr_t>(c.O) & 15) == 0 && c.F % (c.out_bf16 ? 8 : 4) == 0) ? 1 : 0;
  const int smem = smem_of(kind, s);
  if (smem > kMaxSmem) return fail(NK_ERR_NO_SCHEDULE, "conv schedule needs %d bytes of shared memory", smem);
  int grid = sms * ctas_per_sm(kind, s);
  grid = grid / CL * CL;
  if (grid > p.units * CL) grid = p.units * CL;
  if (grid < CL) grid = CL;
  if (kind == TC_FP8) {
    if (mch == 2) status = launch<TC_FP8, 1, false, true, false, false, 2>(p, grid, smem, st);
    else if (mch == 4) status = launch<TC_FP8, 1, false, true, false, false, 4>(p, grid, smem, st);
    else status = launch<TC_FP8, 1, false, true>(p, grid, smem, st);
  } else if (mch == 2) status = launch<TC_BF16, 1, false, true, false, false, 2>(p, grid, smem, st);
  else if (mch == 4) status = launch<TC_BF16, 1, false, true, false, false, 4>(p, grid, smem, st);
  else if (CL == 2) status = launch<TC_BF16, 2, false, true, true>(p, grid, smem, st);
  else status = launch<TC_BF16, 1, false, true>(p, grid, smem, st);
  if (status != NK_OK || splits == 1) return status;
  SplitReduce r{};
  r.partial = p.partial;
  r.ldp = p.ldp;
  r.splits = splits;
  r.M = M;
  r.N = c.F;
  r.C = c.O;
  r.scm = c.F;
  r.scn = 1;
  r.bias = c.bias;
  r.alpha = (kind == TC_FP8 && !c.scale_i) ? c.alpha : 1.f;
  r.beta = c.beta;
  r.relu = c.relu;
  r.scale_a = c.scale_i;
  r.scale_b = c.scale_w;
  r.ew = c.ew;
  r.out_bf16 = c.out_bf16;
  return splitk_reduce(r, st);
}

}  // namespace nk

// ====================================================================== grouped
// linalg.batch_matmul generalised to G independent GEMMs of uneven shapes, all
// in one persistent launch: a device table holds each group's shape, output
// and TMA descriptors, and a prefix sum of tiles per group lets every CTA map
// its running unit index to (group, tile).  A plan also holds the group of
// every unit (one load); a launch from a caller's workspace searches the
// prefix sums instead.  Groups are ordered by decreasing K so the longest
// tiles start first.
struct nk_grouped_plan {
  void* dev = nullptr;     // device table (owned when built by nk_grouped_plan_create)
  int* umap = nullptr;     // [units] group of each unit (plans only)
  bool owned = false;
  bool pair = false;       // 256-row tiles on CTA pairs (cta_group::2)
  bool ep8 = false;        // GEMM groups on one CTA per SM: eight epilogue warps
  bool conv = false;       // groups are convolutions (implicit GEMM, per-tap loads)
  int units = 0;
  int grid = 0;
  int smem = 0;
  nk::TcParams p;
};

namespace nk {
namespace {

// One persistent launch of a grouped GEMM plan: CTA pairs or one CTA per
// tile, with eight epilogue warps when a CTA has the SM to itself.
nk_status run_grouped_gemm(const nk_grouped_plan& plan, cudaStream_t st) {
  if (plan.pair) {
    if (plan.ep8) return launch<TC_BF16, 2, true, false, true, false, 1, true>(plan.p, plan.grid, plan.smem, st);
    return launch<TC_BF16, 2, true, false, true>(plan.p, plan.grid, plan.smem, st);
  }
  if (plan.ep8) return launch<TC_BF16, 1, true, false, false, false, 1, true>(plan.p, plan.grid, plan.smem, st);
  return launch<TC_BF16, 1, true>(plan.p, plan.grid, plan.smem, st);
}

size_t grouped_bytes(int G) {
  size_t maps = (size_t)G * 2 * sizeof(CUtensorMap);
  size_t descs = (size_t)G * sizeof(GroupDesc);
  size_t starts = (size_t)(G + 1) * sizeof(int);
  size_t cmaps = (size_t)G * sizeof(CUtensorMap);   // C maps of the TMA-store epilogue (GEMM groups)
  return maps + ((descs + 127) / 128 * 128) + ((starts + 127) / 128 * 128) + cmaps;
}

nk_schedule grouped_schedule(const nk_schedule* user) {
  nk_schedule s{128, 128, 64, 1, 0, 1};
  if (user) {
    if (user->tile_n) s.tile_n = user->tile_n;
    if (user->stages) s.stages = user->stages;
    if (user->cluster) s.cluster = user->cluster;
    if (user->split_k) s.split_k = user->split_k;
    if (user->tile_m) s.tile_m = user->tile_m;
    if (user->tile_k) s.tile_k = user->tile_k;
  }
  if (s.stages == 0) {
    s.stages = 2;
    while (s.stages < 8 && smem_bytes(TC_BF16, s.tile_n, s.stages + 1) <= kMaxSmem) ++s.stages;
  }
  return s;
}

// The built-in tile of a grouped GEMM: 128 x 128 with the deepest ring, or 128
// x 256 with four stages where the groups fill it.  In units of a 64-deep K
// block of a 128 x 256 tile, a 128 x 128 one costs 0.72 (its MMAs are not half
// as long), and the tiles' epilogues 4 and 2.  Measured, 128 x 128 / 128 x 256,
// us: 512 groups of 32 to 2048 222.7 / 189.9, 512 to 1024 75.5 / 69.7, 32 to
// 2048 26.3 / 22.7; 512 groups of 32 to 512 32.1 / 33.8 (stays 128 x 128).
nk_schedule grouped_gemm_schedule(int G, const nk_gemm_group* groups, const nk_schedule* user) {
  if (user && (user->tile_m || user->tile_n || user->tile_k || user->cluster || user->stages || user->split_k))
    return grouped_schedule(user);
  double square = 0, wide = 0;
  for (int g = 0; g < G; ++g) {
    const nk_gemm_group& q = groups[g];
    if (q.M < 1 || q.N < 1 || q.K < 1) continue;   // refused below
    const double tm = (q.M + 127) / 128, kb = (q.K + 63) / 64;
    square += tm * ((q.N + 127) / 128) * (0.72 * kb + 2);
    wide += tm * ((q.N + 255) / 256) * (kb + 4);
  }
  if (wide < square) return nk_schedule{128, 256, 64, 1, 4, 1};
  return grouped_schedule(nullptr);
}

// Fills `host` (grouped_bytes(G) bytes) with the table for a device buffer at
// `dev_base`, and the launch parameters.
nk_status build_grouped(int G, const nk_gemm_group* groups, int precision, const nk_schedule* user,
                        void* dev_base, std::vector<uint8_t>& host, nk_grouped_plan& plan) {
  if (G < 0) return fail(NK_ERR_INVALID_ARG, "negative group count");
  if (G > 0 && !groups) return fail(NK_ERR_INVALID_ARG, "groups is NULL");
  if (precision != NK_PREC_BF16)
    return fail(NK_ERR_UNSUPPORTED, "grouped GEMM runs BF16 operands (NK_PREC_BF16) only");
  const nk_schedule s = grouped_gemm_schedule(G, groups, user);
  // tile_m 128 on one CTA, or tile_m 256 on a CTA pair (each CTA holds its
  // 128 rows of A and half of the B tile)
  const bool pair = s.tile_m == 256 && s.cluster == 2;
  if (s.split_k != 1 || s.tile_n == 512 || !(pair || (s.tile_m == 128 && s.cluster == 1)) ||
      !tc_schedule_valid(TC_BF16, s, 1, 1, 1))
    return fail(NK_ERR_NO_SCHEDULE,
                "grouped schedule needs split_k 1 and tile_m 128 on one CTA or 256 on a CTA pair");
  const int rows = pair ? 2 * kBM : kBM;   // GEMM rows of one unit
  int sms = 0;
  nk_status st = require_device(&sms);
  if (st != NK_OK) return st;
  // A single-row operand's leading dimension is never stepped over; give TMA
  // a legal one (row padded to 16 bytes) whatever the caller passed.
  auto ld_a = [](const nk_gemm_group& q) { return q.M == 1 ? (int64_t)(q.K + 7) / 8 * 8 : q.lda; };
  auto ld_b = [](const nk_gemm_group& q) { return q.N == 1 ? (int64_t)(q.K + 7) / 8 * 8 : q.ldb; };
  auto ld_c = [](const nk_gemm_group& q) { return q.M == 1 ? (int64_t)(q.N + 3) / 4 * 4 : q.ldc; };
  for (int g = 0; g < G; ++g) {
    nk_gemm_group q = groups[g];
    q.lda = ld_a(q); q.ldb = ld_b(q); q.ldc = ld_c(q);
    if (q.M < 1 || q.N < 1 || q.K < 1) return fail(NK_ERR_INVALID_ARG, "group %d has an empty extent", g);
    if (!q.A || !q.Bt || !q.C) return fail(NK_ERR_INVALID_ARG, "group %d has a NULL pointer", g);
    if (q.lda < q.K || q.ldb < q.K || q.ldc < q.N)
      return fail(NK_ERR_INVALID_ARG, "group %d: leading dimension smaller than the row", g);
    if ((q.lda * 2) % 16 || (q.ldb * 2) % 16 || (reinterpret_cast<uintptr_t>(q.A) & 15) ||
        (reinterpret_cast<uintptr_t>(q.Bt) & 15))
      return fail(NK_ERR_MISALIGNED, "group %d: BF16 operands need 16-byte aligned rows", g);
  }
  std::vector<int> order(G);
  for (int g = 0; g < G; ++g) order[g] = g;
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return groups[a].K > groups[b].K; });
  host.assign(grouped_bytes(G), 0);
  CUtensorMap* maps = reinterpret_cast<CUtensorMap*>(host.data());
  const size_t off_desc = (size_t)G * 2 * sizeof(CUtensorMap);
  const size_t off_start = off_desc + ((size_t)G * sizeof(GroupDesc) + 127) / 128 * 128;
  GroupDesc* descs = reinterpret_cast<GroupDesc*>(host.data() + off_desc);
  int* starts = reinterpret_cast<int*>(host.data() + off_start);
  const size_t off_cmap = off_start + ((size_t)(G + 1) * sizeof(int) + 127) / 128 * 128;
  CUtensorMap* cmaps = reinterpret_cast<CUtensorMap*>(host.data() + off_cmap);
  bool cvec = true, cvec32 = true, ctma = true;
  auto fn = encode_fn();
  int64_t total = 0;
  for (int i = 0; i < G; ++i) {
    nk_gemm_group q = groups[order[i]];
    q.lda = ld_a(q); q.ldb = ld_b(q); q.ldc = ld_c(q);
    if ((st = make_kmajor_map(&maps[2 * i], false, q.A, q.M, q.K, q.lda, kBM)) != NK_OK) return st;
    if ((st = make_kmajor_map(&maps[2 * i + 1], false, q.Bt, q.N, q.K, q.ldb, pair ? s.tile_n / 2 : s.tile_n)) !=
        NK_OK)
      return st;
    GroupDesc& d = descs[i];
    d.M = q.M; d.N = q.N; d.K = q.K;
    d.tiles_n = (q.N + s.tile_n - 1) / s.tile_n;
    d.C = q.C;
    d.ldc = q.ldc;
    d.beta = q.accumulate ? 1.f : 0.f;
    d.kblocks = (q.K + 63) / 64;
    starts[i] = (int)total;
    total += (int64_t)((q.M + rows - 1) / rows) * d.tiles_n;
    if (total > INT32_MAX) return fail(NK_ERR_UNSUPPORTED, "too many tiles");
    cvec = cvec && ((reinterpret_cast<uintptr_t>(q.C) & 15) == 0) && (q.ldc % 4 == 0);
    cvec32 = cvec32 && ((reinterpret_cast<uintptr_t>(q.C) & 31) == 0) && (q.ldc % 8 == 0);
    // TMA-store epilogue: every group a plain overwrite of a 16-byte aligned C
    // whose rows end on 16-byte boundaries (a TMA store clips the innermost
    // dimension to 16-byte granules only)
    ctma = ctma && fn && !q.accumulate && ((reinterpret_cast<uintptr_t>(q.C) & 15) == 0) && (q.ldc * 4) % 16 == 0 &&
           q.N % 4 == 0;
    if (ctma) {
      cuuint64_t dims[2] = {(cuuint64_t)q.N, (cuuint64_t)q.M};
      cuuint64_t strides[1] = {(cuuint64_t)(q.ldc * 4)};
      cuuint32_t box[2] = {32, 32};
      cuuint32_t es[2] = {1, 1};
      ctma = fn(&cmaps[i], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, q.C, dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    }
  }
  starts[G] = (int)total;
  TcParams& p = plan.p;
  memset(&p, 0, sizeof p);
  p.bn = s.tile_n;
  p.stages = s.stages;
  p.units = (int)total;
  p.splits = 1;
  p.alpha = 1.f;
  p.budget = wait_budget();
  p.c_vec = cvec ? 1 : 0;
  p.c_vec32 = cvec32 ? 1 : 0;
  p.G = G;
  uint8_t* db = static_cast<uint8_t*>(dev_base);
  p.gmaps = reinterpret_cast<const CUtensorMap*>(db);
  p.groups = reinterpret_cast<const GroupDesc*>(db + off_desc);
  p.tile_start = reinterpret_cast<const int*>(db + off_start);
  plan.units = (int)total;
  plan.pair = pair;
  plan.ep8 = ctas_per_sm(TC_BF16, s) == 1;
  plan.smem = smem_of(TC_BF16, s);
  // eight epilogue warps stage through eight boxes (four are budgeted)
  if (plan.ep8 && plan.smem + 4 * kStageBox > kMaxSmem) plan.ep8 = false;
  if (plan.ep8) plan.smem += 4 * kStageBox;
  // a second box per warp where it fits beside the CTAs of the SM
  const int stg = staging_bytes(plan.ep8);
  if (ctma && ctas_per_sm(TC_BF16, s) * (plan.smem + stg) <= kMaxSmem) {
    p.boxes2 = 1;
    plan.smem += stg;
  }
  if (ctma) {
    p.gcmaps = reinterpret_cast<const CUtensorMap*>(db + off_cmap);
    p.c_tma = 1;
  }
  const int CL = pair ? 2 : 1;
  int grid = sms * ctas_per_sm(TC_BF16, s) / CL * CL;
  if (grid > plan.units * CL) grid = plan.units * CL;
  plan.grid = grid < CL ? CL : grid;
  return NK_OK;
}

// Grouped convolutions: each group a linalg.conv_2d_nhwc_hwcf on BF16 NHWC
// input and packed BF16 weights, with its own output tiling (ConvTile), 4-D
// input and 3-D weight maps, bias and ReLU in the device table.
nk_status build_grouped_conv(int G, const nk_conv_group* groups, const nk_schedule* user, void* dev_base,
                             std::vector<uint8_t>& host, nk_grouped_plan& plan) {
  if (G < 0) return fail(NK_ERR_INVALID_ARG, "negative group count");
  if (G > 0 && !groups) return fail(NK_ERR_INVALID_ARG, "groups is NULL");
  const nk_schedule s = grouped_schedule(user);
  if (s.tile_m != 128 || s.cluster != 1 || s.split_k != 1 || s.tile_n == 512 || s.tile_k != 64 ||
      !tc_schedule_valid(TC_BF16, s, 1, 1, 1))
    return fail(NK_ERR_NO_SCHEDULE, "grouped conv schedule needs tile_m 128, tile_k 64, cluster 1, split_k 1");
  int sms = 0;
  nk_status st = require_device(&sms);
  if (st != NK_OK) return st;
  std::vector<TcConv> convs(G);
  std::vector<int> kblocks(G);
  for (int i = 0; i < G; ++i) {
    const nk_conv_group& q = groups[i];
    const nk_tensor &I = q.I, &W = q.W, &O = q.O;
    if (I.rank != 4 || W.rank != 4 || O.rank != 4 || I.dtype != NK_BF16 || W.dtype != NK_BF16 || O.dtype != NK_F32)
      return fail(NK_ERR_UNSUPPORTED, "conv group %d: BF16 NHWC I, packed BF16 W and FP32 NHWC O", i);
    for (int d = 0; d < 2; ++d)
      if (q.stride[d] < 1 || q.dilation[d] < 1) return fail(NK_ERR_INVALID_ARG, "conv group %d: stride, dilation", i);
    for (int d = 0; d < 4; ++d)
      if (q.pad[d] < 0) return fail(NK_ERR_INVALID_ARG, "conv group %d: negative padding", i);
    ConvGeom g{};
    g.n = (int)I.shape[0]; g.h = (int)I.shape[1]; g.w = (int)I.shape[2]; g.c = (int)I.shape[3];
    g.kh = (int)W.shape[0]; g.kw = (int)W.shape[1];
    g.sh = (int)q.stride[0]; g.sw = (int)q.stride[1]; g.dh = (int)q.dilation[0]; g.dw = (int)q.dilation[1];
    g.pt = (int)q.pad[0]; g.pl = (int)q.pad[2];
    const int64_t oh = (g.h + q.pad[0] + q.pad[1] - g.dh * (g.kh - 1) - 1) / g.sh + 1;
    const int64_t ow = (g.w + q.pad[2] + q.pad[3] - g.dw * (g.kw - 1) - 1) / g.sw + 1;
    if (oh < 1 || ow < 1 || g.n < 1 || g.c < 1 || W.shape[3] < 1)
      return fail(NK_ERR_INVALID_ARG, "conv group %d: empty problem", i);
    if (W.shape[2] != g.c) return fail(NK_ERR_INVALID_ARG, "conv group %d: I channels != W channels", i);
    if (O.shape[0] != g.n || O.shape[1] != oh || O.shape[2] != ow || O.shape[3] != W.shape[3])
      return fail(NK_ERR_INVALID_ARG, "conv group %d: O must be [%d,%lld,%lld,%lld]", i, g.n, (long long)oh,
                  (long long)ow, (long long)W.shape[3]);
    if (g.sh > 8 || g.sw > 8) return fail(NK_ERR_UNSUPPORTED, "conv group %d: stride above 8", i);
    g.oh = (int)oh; g.ow = (int)ow;
    g.sin_n = I.stride[0]; g.sin_h = I.stride[1]; g.sin_w = I.stride[2];
    const int64_t ldw = W.stride[1], sF = W.stride[3];
    if (I.stride[3] != 1 || W.stride[2] != 1 || ldw < g.c || ldw % 8 || W.stride[0] != W.shape[1] * ldw ||
        sF % 8 || sF < W.shape[0] * W.shape[1] * ldw)
      return fail(NK_ERR_UNSUPPORTED, "conv group %d: I needs unit channel stride, W the packed layout", i);
    if (O.stride[3] != 1 || O.stride[2] != O.shape[3] || O.stride[1] != O.shape[2] * O.stride[2] ||
        O.stride[0] != O.shape[1] * O.stride[1])
      return fail(NK_ERR_UNSUPPORTED, "conv group %d: O must be contiguous NHWC", i);
    if ((g.sin_w * 2) % 16 || (g.sin_h * 2) % 16 || (g.sin_n * 2) % 16 ||
        (reinterpret_cast<uintptr_t>(I.ptr) & 15) || (reinterpret_cast<uintptr_t>(W.ptr) & 15))
      return fail(NK_ERR_MISALIGNED, "conv group %d: operands need 16-byte aligned bases and rows", i);
    if ((int64_t)g.n * g.oh * g.ow > INT32_MAX) return fail(NK_ERR_UNSUPPORTED, "conv group %d: too large", i);
    TcConv& c = convs[i];
    c.kind = TC_BF16;
    c.I = I.ptr; c.sI_n = g.sin_n; c.sI_h = g.sin_h; c.sI_w = g.sin_w;
    c.Wt = W.ptr; c.ldw = ldw; c.sW_f = sF;
    c.g = g;
    c.F = (int)W.shape[3];
    c.O = static_cast<float*>(O.ptr);
    kblocks[i] = g.kh * g.kw * ((g.c + 63) / 64);
  }
  std::vector<int> order(G);
  for (int g = 0; g < G; ++g) order[g] = g;
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return kblocks[a] > kblocks[b]; });
  host.assign(grouped_bytes(G), 0);
  CUtensorMap* maps = reinterpret_cast<CUtensorMap*>(host.data());
  const size_t off_desc = (size_t)G * 2 * sizeof(CUtensorMap);
  const size_t off_start = off_desc + ((size_t)G * sizeof(GroupDesc) + 127) / 128 * 128;
  GroupDesc* descs = reinterpret_cast<GroupDesc*>(host.data() + off_desc);
  int* starts = reinterpret_cast<int*>(host.data() + off_start);
  bool cvec = true;
  int64_t total = 0;
  for (int i = 0; i < G; ++i) {
    const int gi = order[i];
    const TcConv& c = convs[gi];
    const ConvTile t = choose_conv_tile(c.g, TC_BF16);
    if ((st = make_conv_maps(&maps[2 * i], &maps[2 * i + 1], c, t, s.tile_n)) != NK_OK) return st;
    GroupDesc& d = descs[i];
    d.M = c.g.n * c.g.oh * c.g.ow;
    d.N = c.F;
    d.K = c.g.kh * c.g.kw * c.g.c;
    d.tiles_n = (c.F + s.tile_n - 1) / s.tile_n;
    d.C = c.O;
    d.ldc = c.F;
    d.beta = groups[gi].accumulate ? 1.f : 0.f;
    d.kblocks = kblocks[gi];
    d.bias = groups[gi].bias;
    d.relu = groups[gi].relu;
    d.cv = t;
    starts[i] = (int)total;
    total += (int64_t)t.tiles_w * t.tiles_h * ((c.g.n + t.NB - 1) / t.NB) * d.tiles_n;
    if (total > INT32_MAX) return fail(NK_ERR_UNSUPPORTED, "too many tiles");
    cvec = cvec && ((reinterpret_cast<uintptr_t>(c.O) & 15) == 0) && (c.F % 4 == 0);
  }
  starts[G] = (int)total;
  TcParams& p = plan.p;
  memset(&p, 0, sizeof p);
  p.bn = s.tile_n;
  p.stages = s.stages;
  p.units = (int)total;
  p.splits = 1;
  p.alpha = 1.f;
  p.budget = wait_budget();
  p.c_vec = cvec ? 1 : 0;
  p.G = G;
  uint8_t* db = static_cast<uint8_t*>(dev_base);
  p.gmaps = reinterpret_cast<const CUtensorMap*>(db);
  p.groups = reinterpret_cast<const GroupDesc*>(db + off_desc);
  p.tile_start = reinterpret_cast<const int*>(db + off_start);
  plan.units = (int)total;
  plan.pair = false;
  plan.conv = true;
  plan.smem = smem_of(TC_BF16, s);
  int grid = sms * ctas_per_sm(TC_BF16, s);
  if (grid > plan.units) grid = plan.units;
  plan.grid = grid < 1 ? 1 : grid;
  return NK_OK;
}

}  // namespace
}  // namespace nk

using namespace nk;

extern "C" {

nk_status nk_grouped_workspace_size(int32_t G, const nk_gemm_group* groups, int32_t precision,
                                    const nk_schedule* sched, size_t* bytes) {
  (void)groups; (void)precision; (void)sched;
  if (!bytes) return fail(NK_ERR_INVALID_ARG, "bytes is NULL");
  if (G < 0) return fail(NK_ERR_INVALID_ARG, "negative group count");
  *bytes = grouped_bytes(G);
  return NK_OK;
}

namespace nk {
namespace {
// The group of every unit, from the tile prefix sums of the host table.
nk_status attach_unit_map(nk_grouped_plan& plan, const std::vector<uint8_t>& host, int G) {
  if (plan.units <= 0) return NK_OK;
  const size_t off_start = (size_t)G * 2 * sizeof(CUtensorMap) + ((size_t)G * sizeof(GroupDesc) + 127) / 128 * 128;
  const int* starts = reinterpret_cast<const int*>(host.data() + off_start);
  std::vector<int> m((size_t)plan.units);
  int g = 0;
  for (int u = 0; u < plan.units; ++u) {
    while (g + 1 < G && starts[g + 1] <= u) ++g;
    m[(size_t)u] = g;
  }
  cudaError_t e = cudaMalloc(&plan.umap, m.size() * sizeof(int));
  if (e != cudaSuccess) return cuda_fail(e, "cudaMalloc(unit map)");
  e = cudaMemcpy(plan.umap, m.data(), m.size() * sizeof(int), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) { cudaFree(plan.umap); plan.umap = nullptr; return cuda_fail(e, "cudaMemcpy(unit map)"); }
  plan.p.unit_group = plan.umap;
  return NK_OK;
}
}  // namespace
}  // namespace nk

nk_status nk_grouped_plan_create(int32_t G, const nk_gemm_group* groups, int32_t precision,
                                 const nk_schedule* sched, nk_grouped_plan** out) {
  nk::NvtxRange nvtx_range_("nk_grouped_plan_create");
  if (!out) return fail(NK_ERR_INVALID_ARG, "plan is NULL");
  *out = nullptr;
  auto* plan = new nk_grouped_plan();
  void* dev = nullptr;
  const size_t bytes = grouped_bytes(G);
  cudaError_t e = cudaMalloc(&dev, bytes > 0 ? bytes : 1);
  if (e != cudaSuccess) { delete plan; return cuda_fail(e, "cudaMalloc(grouped plan)"); }
  std::vector<uint8_t> host;
  nk_status s = build_grouped(G, groups, precision, sched, dev, host, *plan);
  if (s == NK_OK && bytes) {
    e = cudaMemcpy(dev, host.data(), bytes, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) s = cuda_fail(e, "cudaMemcpy(grouped plan)");
  }
  if (s == NK_OK) s = nk::attach_unit_map(*plan, host, G);
  if (s != NK_OK) { cudaFree(dev); delete plan; return s; }
  plan->dev = dev;
  plan->owned = true;
  *out = plan;
  return NK_OK;
}

nk_status nk_conv2d_grouped_plan_create(int32_t G, const nk_conv_group* groups, const nk_schedule* sched,
                                        nk_grouped_plan** out) {
  nk::NvtxRange nvtx_range_("nk_conv2d_grouped_plan_create");
  if (!out) return fail(NK_ERR_INVALID_ARG, "plan is NULL");
  *out = nullptr;
  auto* plan = new nk_grouped_plan();
  void* dev = nullptr;
  const size_t bytes = grouped_bytes(G);
  cudaError_t e = cudaMalloc(&dev, bytes > 0 ? bytes : 1);
  if (e != cudaSuccess) { delete plan; return cuda_fail(e, "cudaMalloc(grouped conv plan)"); }
  std::vector<uint8_t> host;
  nk_status s = build_grouped_conv(G, groups, sched, dev, host, *plan);
  if (s == NK_OK && bytes) {
    e = cudaMemcpy(dev, host.data(), bytes, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) s = cuda_fail(e, "cudaMemcpy(grouped conv plan)");
  }
  if (s == NK_OK) s = nk::attach_unit_map(*plan, host, G);
  if (s != NK_OK) { cudaFree(dev); delete plan; return s; }
  plan->dev = dev;
  plan->owned = true;
  *out = plan;
  return NK_OK;
}

nk_status nk_grouped_plan_run(const nk_grouped_plan* plan, void* stream) {
  nk::NvtxRange nvtx_range_("nk_grouped_plan_run");
  if (!plan) return fail(NK_ERR_INVALID_ARG, "plan is NULL");
  if (plan->units == 0) return NK_OK;
  if (plan->conv)
    return launch<TC_BF16, 1, true, true>(plan->p, plan->grid, plan->smem, static_cast<cudaStream_t>(stream));
  return run_grouped_gemm(*plan, static_cast<cudaStream_t>(stream));
}

nk_status nk_grouped_plan_destroy(nk_grouped_plan* plan) {
  if (!plan) return NK_OK;
  if (plan->owned && plan->dev) cudaFree(plan->dev);
  if (plan->umap) cudaFree(plan->umap);
  delete plan;
  return NK_OK;
}

nk_status nk_batch_matmul_grouped(int32_t G, const nk_gemm_group* groups, int32_t precision,
                                  const nk_schedule* sched, void* ws, size_t ws_bytes, void* stream) {
  nk::NvtxRange nvtx_range_("nk_batch_matmul_grouped");
  const size_t bytes = grouped_bytes(G);
  if (G > 0 && (!ws || ws_bytes < bytes))
    return fail(NK_ERR_WORKSPACE, "grouped GEMM needs %zu bytes of workspace", bytes);
  if (ws && (reinterpret_cast<uintptr_t>(ws) & 127))
    return fail(NK_ERR_MISALIGNED, "grouped workspace must be 128-byte aligned");
  nk_grouped_plan plan;
  std::vector<uint8_t> host;
  nk_status s = build_grouped(G, groups, precision, sched, ws, host, plan);
  if (s != NK_OK || plan.units == 0) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaMemcpyAsync(ws, host.data(), bytes, cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpyAsync(grouped table)");
  // a pageable source is staged before cudaMemcpyAsync returns, so `host` may go
  return run_grouped_gemm(plan, st);
}

}  // extern "C"
