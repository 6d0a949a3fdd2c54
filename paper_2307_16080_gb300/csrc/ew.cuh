// ew.cuh -- fused elementwise programs (the nk_ew_program of nk.h) as the
// kernels see them, and the per-element interpreter they share.
//
// A program folds the linalg.generic loops that a lowering leaves around a
// contraction -- the bias-add loop of the lowered torch.nn.Linear (Sec. 2.1.2
// Listing "listing1") and the elementwise product of the GPUModule kernel
// (Sec. 3.1 Listing "gpumodules") -- into the kernel that produces (epilogue)
// or reads (prologue) the tensor.  Tensor operands share the layout of the
// tensor the program runs over, so an element's offset from that tensor's
// base also locates its operands.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/nk.h"

namespace nk {

constexpr int kEwMax = NK_EW_MAX;

struct EwProg {
  int n;                    // 0 = no program
  int op[kEwMax];
  float a[kEwMax], b[kEwMax];
  const float* t[kEwMax];   // MUL / ADD operands (offset 0 = the tensor's base)
};

// The same program with every tensor operand moved by `off` elements (a
// kernel that sees a sub-range of the tensor, e.g. one filter tap).
inline EwProg ew_shift(EwProg e, int64_t off) {
  for (int i = 0; i < e.n; ++i)
    if (e.t[i]) e.t[i] += off;
  return e;
}

#ifdef __CUDACC__
// The steps below are branch-free: CUDA's erfcf and its IEEE division take
// data-dependent branches, which keep a warp's independent elements from
// overlapping (measured per warp and element, one warp per scheduler, eight
// elements in flight: GELU with erfcf 141 cycles, x / (1 + e) with the
// division 105, tanhf 28, expf 17).

// n / d for d in [1, 2^93]: the hardware reciprocal and one residual correction
// of the quotient (Markstein, "Computation of elementary functions on the IBM
// RISC System/6000", 1990), which leaves the rounding of an exact division (to
// 2^-44).  Where an infinite n makes the residual a NaN, and for a zero n, whose
// sign it would lose, the uncorrected quotient stands.
static __device__ __forceinline__ float ew_div(float n, float d) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
  const float q = n * r;
  const float c = fmaf(r, fmaf(-d, q, n), q);
  return fabsf(c) > 0.f ? c : q;
}
// y * sigmoid(u) = y / (1 + e^-u): three roundings, as with an IEEE division.
// (y e^u / (1 + e^u) for every u < 0 has a fourth: the worst relative error of
// SiLU was 2.5e-7 that way, on 600 thousand values, and is under 2.4e-7.)
// Below -64 1 + e^-u is e^-u in FP32, and y e^u is the quotient with two; it
// also keeps the results below -88.7 that a division by infinity loses (the
// 1.4 above that, where e^u is subnormal, to 5e-7).
static __device__ __forceinline__ float ew_logistic(float y, float u) {
  const bool low = u < -64.f;
  const float e = expf(low ? u : -u);
  return ew_div(low ? y * e : y, low ? 1.f : 1.f + e);
}

// x * Phi(x).  With a = |x|, Phi(-a) = exp(-a^2 / 2) R(a), where R is half the
// scaled complementary error function erfcx(a / sqrt 2) -- smooth and without
// cancellation, so small results for negative x keep their relative accuracy.
// R is a degree-9 polynomial in (a - 3) / (a + 3) (the change of variable of
// Shepherd & Laframboise, "Chebyshev approximation of (1 + 2x) exp(x^2)
// erfc x in 0 <= x < inf", 1981), fitted here to R on [0, 14.3] with a
// relative error of 9e-9.  exp(-a^2 / 2) takes the rounding error of a^2
// along and reduces the exponent in two parts; 2^n is applied as 2^(n+60)
// 2^-60 so that results below the smallest normal number round once.
//
// Two elements at a time on the packed FP32 instructions (one issue slot for
// two lanes' worth of FMA, each half rounded as the scalar instruction is):
// an epilogue warp is bound by what it can issue.  Bias + GELU on 4096 x 4096 x
// 1024 BF16 (128 x 256 tiles): 53.3 us scalar, 46.6 us packed.
struct f2 {
  uint64_t v;
};
static __device__ __forceinline__ f2 f2_make(float lo, float hi) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
  return r;
}
static __device__ __forceinline__ f2 f2_set(float x) { return f2_make(x, x); }
static __device__ __forceinline__ void f2_get(f2 a, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v));
}
static __device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
static __device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
static __device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}

static __device__ __forceinline__ void ew_gelu2(float& x0, float& x1) {
  const float a0 = fminf(fabsf(x0), 16.f), a1 = fminf(fabsf(x1), 16.f);   // Phi(-16) is 0 in FP32
  const f2 a = f2_make(a0, a1);
  float t0, t1, r0, r1;
  f2_get(f2_add(a, f2_set(3.f)), t0, t1);
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(t0));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r1) : "f"(t1));
  const f2 q = f2_mul(f2_add(a, f2_set(-3.f)), f2_make(r0, r1));
  f2 p = f2_set(5.336296453606337e-05f);
  p = f2_fma(p, q, f2_set(0.00011522331624291837f));
  p = f2_fma(p, q, f2_set(-0.00033920127316378057f));
  p = f2_fma(p, q, f2_set(-0.0009834759403020144f));
  p = f2_fma(p, q, f2_set(0.00290445564314723f));
  p = f2_fma(p, q, f2_set(0.006131994072347879f));
  p = f2_fma(p, q, f2_set(-0.04621327295899391f));
  p = f2_fma(p, q, f2_set(0.12322503328323364f));
  p = f2_fma(p, q, f2_set(-0.20640261471271515f));
  p = f2_fma(p, q, f2_set(0.12151394784450531f));
  const f2 s = f2_mul(a, a);
  const f2 ms = f2_make(-a0, -a1);
  const f2 me = f2_fma(a, ms, s);                     // a^2 = s - me
  constexpr float L = -0.72134752044448170f;          // -log2(e) / 2, and what FP32 drops of it
  constexpr float LL = (float)(-0.72134752044448170368 - (double)L);
  const f2 big = f2_fma(s, f2_set(L), f2_set(12582912.f));   // 1.5 * 2^23 + n, n = rint(s L)
  const f2 mn = f2_fma(big, f2_set(-1.f), f2_set(12582912.f));
  f2 f = f2_fma(s, f2_set(L), mn);
  f = f2_fma(s, f2_set(LL), f);
  f = f2_fma(me, f2_set(-L), f);
  float f0, f1, e0, e1, b0, b1;
  f2_get(f, f0, f1);
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(f0));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(f1));
  f2_get(big, b0, b1);
  const f2 sc = f2_make(__int_as_float((__float_as_int(b0) << 23) + ((127 + 60) << 23)),   // 2^(n + 60)
                        __int_as_float((__float_as_int(b1) << 23) + ((127 + 60) << 23)));
  p = f2_mul(f2_mul(f2_mul(f2_make(e0, e1), p), sc), f2_set(0x1p-60f));
  // x Phi(x): x p for x < 0, x - x p otherwise (1 - Phi(6) is under half an ulp of 1)
  const f2 y = f2_fma(f2_make(-fabsf(x0), -fabsf(x1)), p, f2_make(fmaxf(x0, 0.f), fmaxf(x1, 0.f)));
  float y0, y1;
  f2_get(y, y0, y1);
  x0 = x0 <= 6.f && x0 != 0.f ? y0 : x0;   // a NaN and the sign of a zero stay
  x1 = x1 <= 6.f && x1 != 0.f ? y1 : x1;
}
static __device__ __forceinline__ float ew_gelu(float x) {
  float y = 0.f;
  ew_gelu2(x, y);
  return x;
}

// One step without a tensor operand, FP32 throughout.  The tanh form of GELU
// is x sigmoid(2u): (1 + tanh u) / 2 without its cancellation.
static __device__ __forceinline__ float ew_step(int op, float x, float a, float b) {
  switch (op) {
    case NK_EW_AFFINE: return __fmaf_rn(a, x, b);
    case NK_EW_RELU: return (x > 0.f || x != x) ? x : 0.f;
    case NK_EW_GELU: return ew_gelu(x);
    case NK_EW_GELU_TANH: {
      const float u = 0.79788456080286536f * fmaf(0.044715f * x, x * x, x);
      return ew_logistic(x, 2.f * u);
    }
    case NK_EW_SILU: return ew_logistic(x, x);
    case NK_EW_SIGMOID: return ew_logistic(1.f, x);
    case NK_EW_TANH: return tanhf(x);
    case NK_EW_CLAMP: return x < a ? a : (x > b ? b : x);
    default: return x;
  }
}

// Runs program `e` on value x of the element at offset `off`.  Kept out of
// line: the unrolled loads and epilogues call it per element only when a
// program is present, and the plain paths carry no extra code.
static __device__ __noinline__ float ew_run(const EwProg& e, float x, int64_t off) {
  for (int i = 0; i < e.n; ++i) {
    const float a = e.a[i], b = e.b[i];
    switch (e.op[i]) {
      case NK_EW_MUL: x = __fmul_rn(x, e.t[i][off]); break;
      case NK_EW_ADD: x = __fadd_rn(x, e.t[i][off]); break;
      default: x = ew_step(e.op[i], x, a, b);
    }
  }
  return x;
}

// One operation of a program on V values in registers; t: the tensor operand's
// first n elements beside them (read only there).  An epilogue has one or two
// warps per scheduler, so latency is what bounds a program: V independent
// elements per dispatch keep a warp issuing.
template <int V>
static __device__ __forceinline__ void ew_op(int op, float a, float b, const float* t, float (&x)[V], int n) {
  switch (op) {
    case NK_EW_MUL:
    case NK_EW_ADD: {
      float y[V];
      if (n >= V && (reinterpret_cast<uintptr_t>(t) & 15) == 0) {
#pragma unroll
        for (int j = 0; j < V; j += 4) {
          const float4 q = *reinterpret_cast<const float4*>(t + j);
          y[j] = q.x; y[j + 1] = q.y; y[j + 2] = q.z; y[j + 3] = q.w;
        }
      } else {
#pragma unroll
        for (int j = 0; j < V; ++j) y[j] = j < n ? t[j] : 0.f;
      }
#pragma unroll
      for (int j = 0; j < V; ++j) x[j] = op == NK_EW_MUL ? __fmul_rn(x[j], y[j]) : __fadd_rn(x[j], y[j]);
      break;
    }
#define NK_EW_CASE(OP)                                                            \
  case OP:                                                                        \
    _Pragma("unroll") for (int j = 0; j < V; ++j) x[j] = ew_step(OP, x[j], a, b); \
    break;
    NK_EW_CASE(NK_EW_AFFINE)
    NK_EW_CASE(NK_EW_RELU)
    case NK_EW_GELU:
#pragma unroll
      for (int j = 0; j < V; j += 2) ew_gelu2(x[j], x[j + 1]);
      break;
    NK_EW_CASE(NK_EW_GELU_TANH)
    NK_EW_CASE(NK_EW_SILU)
    NK_EW_CASE(NK_EW_SIGMOID)
    NK_EW_CASE(NK_EW_TANH)
    NK_EW_CASE(NK_EW_CLAMP)
#undef NK_EW_CASE
    default: break;
  }
}

// Runs program `e` on the 32 values v, elements at offsets off0 .., of which
// the first n exist (n = 0: v is padding and stays undefined).  Inline, for
// the kernel variants that are instantiated for programs: everything stays in
// registers, and opcodes and coefficients come from the parameter bank.
static __device__ __forceinline__ void ew_regs(const EwProg& e, float (&v)[32], int n, int64_t off0) {
#pragma unroll 1
  for (int i = 0; i < e.n; ++i) ew_op<32>(e.op[i], e.a[i], e.b[i], e.t[i] + off0, v, n);
}

// The same out of line on a buffer (16-byte aligned, all 32 floats defined),
// for the epilogues that have no variant of their own: they stage a 32-column
// segment in a local buffer, call this, then store.  The program reads its
// operands (which may alias the output) before the store, and the plain
// epilogue keeps no call in its unrolled body.  Eight elements at a time: a
// callee's registers count for every kernel that calls it, and more would take
// the second CTA of an SM away from the plain variants.
static __device__ __noinline__ void ew_op_buf(int op, float a, float b, const float* t, float* buf, int n) {
#pragma unroll 1
  for (int c = 0; c < n; c += 8) {
    float x[8];
#pragma unroll
    for (int j = 0; j < 8; j += 4) {
      const float4 q = *reinterpret_cast<const float4*>(buf + c + j);
      x[j] = q.x; x[j + 1] = q.y; x[j + 2] = q.z; x[j + 3] = q.w;
    }
    ew_op<8>(op, a, b, t + c, x, n - c);
#pragma unroll
    for (int j = 0; j < 8; j += 4) *reinterpret_cast<float4*>(buf + c + j) = make_float4(x[j], x[j + 1], x[j + 2], x[j + 3]);
  }
}
static __device__ __forceinline__ void ew_apply(const EwProg& e, float* buf, int n, int64_t off0) {
#pragma unroll 1
  for (int i = 0; i < e.n; ++i) ew_op_buf(e.op[i], e.a[i], e.b[i], e.t[i] + off0, buf, n);
}

// v[j] += bias[j] for 32 columns that all exist: eight 16-byte loads (the same
// for every lane) where the bias allows them, 32 scalar ones else.
__device__ __forceinline__ void add_bias32(const float* bias, float (&v)[32]) {
  if ((reinterpret_cast<uintptr_t>(bias) & 15) == 0) {
#pragma unroll
    for (int j = 0; j < 32; j += 4) {
      const float4 b = *reinterpret_cast<const float4*>(bias + j);
      v[j] += b.x; v[j + 1] += b.y; v[j + 2] += b.z; v[j + 3] += b.w;
    }
  } else {
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] += bias[j];
  }
}

// 32-byte stores (one whole L2 sector per thread; the address must be
// 32-byte aligned).  The epilogues write one output row per lane, so a warp
// store touches 32 rows: with 16-byte stores each row's sector arrives in
// two halves, with these in one piece, and the L2 sees half the requests.
__device__ __forceinline__ void st_v8_f32(float* p, float a0, float a1, float a2, float a3, float a4, float a5,
                                          float a6, float a7) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(a0), "f"(a1), "f"(a2),
               "f"(a3), "f"(a4), "f"(a5), "f"(a6), "f"(a7)
               : "memory");
}
__device__ __forceinline__ void st_v8_b32(void* p, const uint32_t* w) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(w[0]), "r"(w[1]), "r"(w[2]),
               "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
               : "memory");
}
// 32 consecutive FP32 values to a 32-byte aligned row segment.
__device__ __forceinline__ void store32_f32_v8(float* dst, const float* v) {
#pragma unroll
  for (int j = 0; j < 32; j += 8) st_v8_f32(dst + j, v[j], v[j + 1], v[j + 2], v[j + 3], v[j + 4], v[j + 5], v[j + 6], v[j + 7]);
}

// BF16 outputs (a convolution whose result feeds the next layer directly):
// the epilogue computes in FP32 as for an FP32 output, then rounds each
// value to BF16 with round-to-nearest-even (CUDA's conversion intrinsic).
// 32 consecutive values to a 16-byte aligned row segment: four 16-byte
// stores of eight BF16 each.
__device__ __forceinline__ void store32_bf16(__nv_bfloat16* dst, const float* v) {
#pragma unroll
  for (int j = 0; j < 32; j += 8) {
    __nv_bfloat162 h[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) h[e] = __floats2bfloat162_rn(v[j + 2 * e], v[j + 2 * e + 1]);
    *reinterpret_cast<uint4*>(dst + j) = *reinterpret_cast<const uint4*>(h);
  }
}
// The same to a 32-byte aligned segment in two 32-byte stores.
__device__ __forceinline__ void store32_bf16_v8(__nv_bfloat16* dst, const float* v) {
#pragma unroll
  for (int j = 0; j < 32; j += 16) {
    __nv_bfloat162 h[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) h[e] = __floats2bfloat162_rn(v[j + 2 * e], v[j + 2 * e + 1]);
    st_v8_b32(dst + j, reinterpret_cast<const uint32_t*>(h));
  }
}
#endif

}  // namespace nk
