// ivhd_gelu.cuh -- GELU(x) = x Phi(x) in FP32 without branches, two values at a time.
//
// Phi(-a) = erfc(a / sqrt 2) / 2 for a = |x|, and erfc(z) = exp(-z^2) erfcx(z), so
//
//   GELU(x) = max(x, 0) - a/2 * 2^( -a^2 log2(e)/2 + p(a) ),   p(a) = log2 erfcx(a / sqrt 2).
//
// p is smooth (0 at a = 0, about -2.9 at a = 5.7); a polynomial a (c1 + .. + c9 a^8)
// was fitted to it on [0, 4 sqrt 2] by linear programming (minimax of the error
// it causes in GELU and Phi: 2.4e-9) against erfcx in 64 bits; beyond that
// range p keeps its end value, where 2^(..) is below 1e-8.  Nothing cancels for
// x < 0, unlike 0.5 x (1 + erf(x / sqrt 2)) in FP32.  Against 64 bits on the
// GPU, uniform x, norm-wise (the erff form in brackets): [-12, 12] 8.5e-9
// (1.2e-8), [-4, 4] 2.3e-8 (3.6e-8), [-1, 1] 3.5e-8 (4.0e-8), [-6, -3] 1.8e-6 (5.4e-5).
// x = +inf gives +inf, -inf gives 0, NaN gives NaN.
// Cost: eight packed FMAs and one exponential a value and half; the erff form
// took both sides of a branch for most warps.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace ivhd {

// Two FP32 values in one 64-bit register: the packed FMA pipe of sm_100 and later.
struct F2 {
  uint64_t v;
};
__device__ __forceinline__ F2 f2(float a, float b) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 f2_get(F2 a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
  return r;
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 f2_same(float a) { return f2(a, a); }
__device__ __forceinline__ float ex2(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// 2^(-a^2 log2(e)/2 + p(a)) = erfc(a / sqrt 2) = 2 Phi(-a) for a = |x|, both
// values; t = min(a, 4 sqrt 2).
__device__ __forceinline__ float2 erfc_half(F2 x, F2& t) {
  const float2 s = f2_get(x);
  const F2 a = f2(fabsf(s.x), fabsf(s.y));
  t = f2(fminf(fabsf(s.x), 5.65685425f), fminf(fabsf(s.y), 5.65685425f));
  F2 p = f2_same(4.474227069e-07f);
  p = f2_fma(p, t, f2_same(-8.659556443e-06f));
  p = f2_fma(p, t, f2_same(6.996341108e-05f));
  p = f2_fma(p, t, f2_same(-2.698139870e-04f));
  p = f2_fma(p, t, f2_same(-8.659691048e-06f));
  p = f2_fma(p, t, f2_same(6.952732336e-03f));
  p = f2_fma(p, t, f2_same(-5.244524777e-02f));
  p = f2_fma(p, t, f2_same(2.621284127e-01f));
  p = f2_fma(p, t, f2_same(-1.151104450e+00f));
  const F2 q = f2_fma(f2_mul(a, f2_same(-0.72134752044448170f)), a, f2_mul(p, t));
  const float2 e = f2_get(q);
  return make_float2(ex2(e.x), ex2(e.y));
}

// GELU of both values.  The factor a stops at the end of the polynomial's range
// too, where the product is below 4e-8 and falling: an infinite x does not meet
// the exponential's zero as inf * 0.
__device__ __forceinline__ float2 gelu2(F2 x) {
  F2 t;
  const float2 e = erfc_half(x, t), s = f2_get(x);
  return f2_get(f2_fma(f2_mul(t, f2_same(-0.5f)), f2(e.x, e.y), f2(fmaxf(s.x, 0.f), fmaxf(s.y, 0.f))));
}

// GELU'(x) = Phi(x) + x phi(x) of both values.
__device__ __forceinline__ float2 gelu_grad2(F2 x) {
  F2 t;
  const float2 e = erfc_half(x, t), s = f2_get(x);
  // Phi = 1/2 + copysign(1/2 - Phi(-a), x)
  const float2 c = f2_get(f2_fma(f2(e.x, e.y), f2_same(-0.5f), f2_same(0.5f)));
  const F2 cdf = f2_add(f2(copysignf(c.x, s.x), copysignf(c.y, s.y)), f2_same(0.5f));
  const float2 g = f2_get(f2_mul(f2_mul(x, f2_same(-0.72134752044448170f)), x));
  const F2 pdf = f2_mul(f2(ex2(g.x), ex2(g.y)), f2_same(0.39894228040143268f));
  return f2_get(f2_fma(x, pdf, cdf));
}

}  // namespace ivhd
