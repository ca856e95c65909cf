// Device helpers shared by the fused MLP forward kernels: paired float32
// arithmetic, bias + GELU + bfloat16 of two activations, ordered score keys.
#pragma once

#include <stdint.h>

#include <cuda_bf16.h>

namespace ktune {

__device__ __forceinline__ int okey_p(float f) {
  const int b = __float_as_int(f);
  return b >= 0 ? b : b ^ 0x7FFFFFFF;
}

// Round-to-nearest-even bfloat16 pair (lo in the low half), one conversion.
__device__ __forceinline__ uint32_t bf2(float lo, float hi) {
  const __nv_bfloat162 b = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t *>(&b);
}

// The paired f32x2 instructions of sm_100 and later: each half one IEEE
// round-to-nearest operation.
__device__ __forceinline__ uint64_t f2pk(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ uint64_t f2fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t f2mul(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t f2add(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// GELU(z) = z (1 + erf(z / sqrt 2)) / 2 with erf from Abramowitz & Stegun,
// Handbook of Mathematical Functions, formula 7.1.28 (Hastings):
//   erf(x) = 1 - (1 + a1 x + a2 x^2 + ... + a6 x^6)^-16 + e(x),  x >= 0,
//   |e(x)| <= 3e-7.
// The bracket's inverse 16th power q is erfc(|x|), so (1 + erf(z / sqrt 2)) / 2
// is 1 - q / 2 for z >= 0 and q / 2 itself for z < 0 (no cancellation for
// negative z).  For z >= 16 the power overflows, q is 0 and GELU(z) = z exactly.
// With float32 arithmetic the result is within 4e-7 max(|z|, 1) of the exact
// GELU (a float64 comparison over a dense grid of [-12, 20]), far below the
// bfloat16 rounding the activation then takes.
// Two GELUs at once, of z = v + bias for both halves.  With o = 1 for z >= 0
// and 0 for z < 0 (one set instruction), |o - q / 2| is both sides in one
// multiply-add, without a select, and the absolute values are operand
// modifiers: 28 cycles of the FMA pipe a pair (a paired instruction takes two),
// which is what bounds the forward kernel.  Returns their
// round-to-nearest-even bfloat16 pair.
__device__ __forceinline__ float ge0(float z) {
  float o;
  asm("set.ge.f32.f32 %0, %1, 0f00000000;" : "=f"(o) : "f"(z));
  return o;
}
__device__ __forceinline__ uint32_t gelu2_bf(float v0, float b0, float v1, float b1) {
  const uint64_t z = f2add(f2pk(v0, v1), f2pk(b0, b1));
  float z0, z1;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(z0), "=f"(z1) : "l"(z));
  const uint64_t x = f2pk(__fmul_rn(fabsf(z0), 0.70710678118654752f),
                          __fmul_rn(fabsf(z1), 0.70710678118654752f));
  uint64_t p = f2fma(f2pk(4.30638e-5f, 4.30638e-5f), x, f2pk(2.765672e-4f, 2.765672e-4f));
  p = f2fma(p, x, f2pk(1.520143e-4f, 1.520143e-4f));
  p = f2fma(p, x, f2pk(9.2705272e-3f, 9.2705272e-3f));
  p = f2fma(p, x, f2pk(4.22820123e-2f, 4.22820123e-2f));
  p = f2fma(p, x, f2pk(7.05230784e-2f, 7.05230784e-2f));
  p = f2fma(p, x, f2pk(1.0f, 1.0f));
  p = f2mul(p, p);
  p = f2mul(p, p);
  p = f2mul(p, p);
  p = f2mul(p, p);
  float p0, p1, q0, q1, t0, t1;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(p0), "=f"(p1) : "l"(p));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(q0) : "f"(p0));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(q1) : "f"(p1));
  const uint64_t t = f2fma(f2pk(q0, q1), f2pk(-0.5f, -0.5f), f2pk(ge0(z0), ge0(z1)));
  asm("mov.b64 {%0, %1}, %2;" : "=f"(t0), "=f"(t1) : "l"(t));
  return bf2(__fmul_rn(z0, fabsf(t0)), __fmul_rn(z1, fabsf(t1)));
}

}  // namespace ktune
