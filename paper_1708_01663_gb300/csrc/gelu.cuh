// GELU and its derivative for the FNO kernels, without a branch and with one
// reciprocal (plus one exponential for the derivative):
//   gelu(x)  = x Phi(x) = (x + |x| erf(|x| / sqrt 2)) / 2
//   gelu'(x) = Phi(x) + x phi(x),  phi(x) = exp(-x^2 / 2) / sqrt(2 pi)
// erf on z >= 0 is the rational form of Abramowitz & Stegun, Handbook of
// Mathematical Functions, 7.1.28 (after Hastings):
//   erf(z) = 1 - (1 + a1 z + a2 z^2 + ... + a6 z^6)^-16,  |error| <= 3e-7,
// with z clamped at 4 (erf(4) = 1 - 1.5e-8), which keeps the 16th power finite.
// In FP32 the 16th power multiplies the polynomial's rounding by 16: the
// evaluated erf is within 2e-6 (the host build of this header is checked
// against std::erf), far below the BF16-split GEMMs' 1.5e-5.
#pragma once
#include <math.h>

namespace cisor {

__host__ __device__ __forceinline__ float gelu_rcp(float p) {
#ifdef __CUDA_ARCH__
  return __fdividef(1.f, p);
#else
  return 1.f / p;
#endif
}

__host__ __device__ __forceinline__ float gelu_exp(float x) {
#ifdef __CUDA_ARCH__
  return __expf(x);
#else
  return expf(x);
#endif
}

// Two values at once: on the device the pair's sums, products and multiply-adds are single packed instructions of
// the sm_100 family (same rounding, half the issue slots; the FNO's row kernels are bound by issue in these
// functions).  The host build computes the halves one by one.
__host__ __device__ __forceinline__ float2 pair_fma(float2 a, float2 b, float2 c) {
#ifdef __CUDA_ARCH__
  return __ffma2_rn(a, b, c);
#else
  return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y));
#endif
}
__host__ __device__ __forceinline__ float2 pair_mul(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
  return __fmul2_rn(a, b);
#else
  return make_float2(a.x * b.x, a.y * b.y);
#endif
}
__host__ __device__ __forceinline__ float2 pair_add(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
  return __fadd2_rn(a, b);
#else
  return make_float2(a.x + b.x, a.y + b.y);
#endif
}
__host__ __device__ __forceinline__ float2 pair_of(float a) { return make_float2(a, a); }
__host__ __device__ __forceinline__ float2 pair_sub(float2 a, float2 b) { return pair_fma(b, pair_of(-1.f), a); }

// erf(z) for z >= 0
__host__ __device__ __forceinline__ float2 erf_pos(float2 z) {
  z = make_float2(fminf(z.x, 4.f), fminf(z.y, 4.f));
  float2 p = pair_fma(pair_of(4.30638e-5f), z, pair_of(2.765672e-4f));
  p = pair_fma(p, z, pair_of(1.520143e-4f));
  p = pair_fma(p, z, pair_of(9.2705272e-3f));
  p = pair_fma(p, z, pair_of(4.22820123e-2f));
  p = pair_fma(p, z, pair_of(7.05230784e-2f));
  p = pair_fma(p, z, pair_of(1.f));
  p = pair_mul(p, p);
  p = pair_mul(p, p);
  p = pair_mul(p, p);
  p = pair_mul(p, p);
  return pair_sub(pair_of(1.f), make_float2(gelu_rcp(p.x), gelu_rcp(p.y)));
}

__host__ __device__ __forceinline__ float2 gelu_f(float2 x) {
  const float2 a = make_float2(fabsf(x.x), fabsf(x.y));
  return pair_mul(pair_of(0.5f), pair_fma(a, erf_pos(pair_mul(a, pair_of(0.70710678118654752f))), x));
}

// both at once (one erf): g = gelu(x), the result gelu'(x)
__host__ __device__ __forceinline__ float2 gelu_and_grad(float2 x, float2& g) {
  const float2 a = make_float2(fabsf(x.x), fabsf(x.y));
  const float2 e = erf_pos(pair_mul(a, pair_of(0.70710678118654752f)));
  g = pair_mul(pair_of(0.5f), pair_fma(a, e, x));
  const float2 h = pair_mul(pair_mul(x, pair_of(-0.5f)), x);
  const float2 phi = pair_fma(make_float2(copysignf(e.x, x.x), copysignf(e.y, x.y)), pair_of(0.5f), pair_of(0.5f));
  return pair_fma(pair_mul(x, pair_of(0.39894228040143268f)), make_float2(gelu_exp(h.x), gelu_exp(h.y)), phi);
}
__host__ __device__ __forceinline__ float2 gelu_grad_f(float2 x) {
  float2 g;
  return gelu_and_grad(x, g);
}

// one value
__host__ __device__ __forceinline__ float erf_pos(float z) { return erf_pos(make_float2(z, z)).x; }
__host__ __device__ __forceinline__ float gelu_f(float x) { return gelu_f(make_float2(x, x)).x; }
__host__ __device__ __forceinline__ float gelu_grad_f(float x) { return gelu_grad_f(make_float2(x, x)).x; }
__host__ __device__ __forceinline__ void gelu_and_grad(float x, float& g, float& gp) {
  float2 g2;
  gp = gelu_and_grad(make_float2(x, x), g2).x;
  g = g2.x;
}

}  // namespace cisor
