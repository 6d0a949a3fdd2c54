// cluster_sum.cuh -- split-K inside a thread-block cluster: the CTAs of a
// cluster each compute one slice of a tile's reduction, leave their FP32
// partial tile in their own shared memory, and each finishes a share of its
// rows, adding the slices in rank order through distributed shared memory.
// Against partial tiles in global memory and a reduce kernel this saves the
// second launch and a round trip of `slices` tiles through L2; the order of
// addition is fixed, so results are the same every run.
#pragma once

#include <stdint.h>

#include "ew.cuh"
#include "tc_ptx.cuh"

namespace nk {

// Partial tile: 128 rows of `bn` floats with a row stride of bn + 4 floats,
// which keeps the 16-byte stores of 32 lanes (one row each) and the row-wise
// reads free of bank conflicts.
__host__ __device__ inline int partial_ld(int bn) { return bn + 4; }
__host__ __device__ inline int partial_bytes(int bn) { return 128 * partial_ld(bn) * (int)sizeof(float); }

// The epilogue of a row of outputs (see nk_epilogue).
struct RowOut {
  float* C;
  int N;                 // columns of C
  const float* bias;
  int bias_on_m, relu;
  float alpha, beta;
};

__device__ __forceinline__ void store_partial32(uint32_t part, int bn, int row, int c0, const float (&v)[32]) {
  const uint32_t at = part + (uint32_t)((row * partial_ld(bn) + c0) * 4);
#pragma unroll
  for (int j = 0; j < 32; j += 4)
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(at + 4u * j), "f"(v[j]), "f"(v[j + 1]), "f"(v[j + 2]),
                 "f"(v[j + 3])
                 : "memory");
}

__device__ __forceinline__ float4 ld_cluster_f4(uint32_t addr) {
  float4 v;   // volatile: in order with the cluster barriers around it
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
  return v;
}

// Four outputs (columns col .. col + 3 of the row at element `off`, row m).
__device__ __forceinline__ void finish4(const RowOut& o, const EwProg& ew, const float (&s)[4], const float (&b)[4],
                                        int64_t off, int m, int col) {
  float x[4];
  float* f = o.C + off + col;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    float y = o.alpha * s[e];
    if (col + e < o.N) {
      if (o.beta != 0.f) y = fmaf(o.beta, f[e], y);
      if (o.bias) y += o.bias_on_m ? __ldg(o.bias + m) : b[e];
      if (o.relu) y = (y > 0.f || y != y) ? y : 0.f;
      if (ew.n) y = ew_run(ew, y, off + col + e);
    }
    x[e] = y;
  }
  if (col + 4 <= o.N && (reinterpret_cast<uintptr_t>(f) & 15) == 0) {
    *reinterpret_cast<float4*>(f) = make_float4(x[0], x[1], x[2], x[3]);
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (col + e < o.N) f[e] = x[e];
  }
}

// Finishes this CTA's 128 / CS rows of the cluster's tile (columns col0 ..):
// every thread takes groups of four columns, U at a time, so that U * CS
// remote loads are in flight.  The slices are added in the order of the reduce
// kernel's shuffle tree (r and r + CS / 2, then halves of that), so both give
// the same bits.  place(row, &off, &m): the output row of tile row `row`
// (element offset, row index), or false for padding.
template <int CS, int U, int THREADS, typename Place>
__device__ __forceinline__ void finish_share(const RowOut& o, const EwProg& ew, uint32_t part, int bn, int crank, int col0,
                                             const Place& place) {
  constexpr int SHARE = 128 / CS;
  const int quads = bn / 4, items = SHARE * quads;
  // bn is 64, 128 or 256 and THREADS a multiple of 64: a thread's columns are
  // the same in every group
  const int c = (int)threadIdx.x % quads * 4, col = col0 + c;
  float b[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) b[e] = o.bias && !o.bias_on_m && col + e < o.N ? __ldg(o.bias + col + e) : 0.f;
  for (int i0 = threadIdx.x; i0 < items; i0 += THREADS * U) {
    float4 q[U][CS];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * THREADS < items ? i0 + u * THREADS : i0;
      const uint32_t at = part + (uint32_t)(((crank * SHARE + i / quads) * partial_ld(bn) + c) * 4);
#pragma unroll
      for (int r = 0; r < CS; ++r) q[u][r] = ld_cluster_f4(ptx::mapa(at, (uint32_t)r));
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * THREADS;
      if (i >= items) break;
      float s[CS][4];
#pragma unroll
      for (int r = 0; r < CS; ++r) { s[r][0] = q[u][r].x; s[r][1] = q[u][r].y; s[r][2] = q[u][r].z; s[r][3] = q[u][r].w; }
#pragma unroll
      for (int h = CS / 2; h >= 1; h /= 2)
#pragma unroll
        for (int r = 0; r < h; ++r)
#pragma unroll
          for (int e = 0; e < 4; ++e) s[r][e] += s[r + h][e];
      int64_t off;
      int m;
      if (col < o.N && place(crank * SHARE + i / quads, off, m)) finish4(o, ew, s[0], b, off, m, col);
    }
  }
}

template <int THREADS, typename Place>
__device__ __forceinline__ void finish_tile(const RowOut& o, const EwProg& ew, uint32_t part, int bn, int cs, int crank,
                                            int col0, const Place& place) {
  if (cs == 2) finish_share<2, 6, THREADS>(o, ew, part, bn, crank, col0, place);
  else if (cs == 4) finish_share<4, 3, THREADS>(o, ew, part, bn, crank, col0, place);
  else finish_share<8, 2, THREADS>(o, ew, part, bn, crank, col0, place);
}

}  // namespace nk
