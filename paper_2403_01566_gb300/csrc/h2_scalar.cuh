// Scalar pieces of the factorisation kernels: conversions between FP64 and
// FP32 by bit operations, reciprocals and the rotation of a Jacobi pair.  No
// shared state, so that they can also be compiled and checked on the host.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

namespace h2 {

// v as FP32 by bit operations (no FP64 instruction), the fraction truncated to
// 23 bits; below FP32's normal range 0, above it the largest exponent.
__device__ __forceinline__ float f32_of_normal(double v) {
  const unsigned hw = (unsigned)__double2hiint(v), lw = (unsigned)__double2loint(v);
  const int a = (int)(hw & 0x7fffffffu) - (896 << 20);
  const unsigned m = a < (1 << 20) ? 0u : ((unsigned)min(a, (255 << 20) - 1) << 3) | (lw >> 29);
  return __uint_as_float((hw & 0x80000000u) | m);
}

// f 2^k as FP64, exactly, by bit operations (f normal or zero)
__device__ __forceinline__ double f64_of_f32_scaled(float f, int k) {
  const unsigned u = __float_as_uint(f);
  const int ef = (int)((u >> 23) & 0xffu);
  if (ef == 0) return 0.0;
  const unsigned hw = (u & 0x80000000u) | ((unsigned)(ef - 127 + 1023 + k) << 20) | ((u & 0x7fffffu) >> 3);
  return __hiloint2double((int)hw, (int)((u & 0x7u) << 29));
}

// 1 / sqrt(v) and 1 / v of a positive v: an FP32 seed x0 of the value scaled
// into [1, 4) ([1, 2)) and one step of third order, about six FP64
// instructions each beside integer ones, where the library functions take
// about thirteen together with their special cases; those of subnormal or
// infinite values, and NaN, are left to them.
__device__ __forceinline__ double rsqrt_pos(double v) {
  const int hi = __double2hiint(v), e = hi >> 20;
  if ((unsigned)(e - 1) >= 0x7feu) return rsqrt(v);
  const int q = (e - 1023) & ~1;  // even exponent
  const double m = __hiloint2double(hi - (q << 20), __double2loint(v));
  const double x0 = f64_of_f32_scaled(rsqrtf(f32_of_normal(m)), 0);
  const double r = fma(-(m * x0), x0, 1.0);
  const double x = fma(x0, r * fma(r, 0.375, 0.5), x0);
  return __hiloint2double(__double2hiint(x) - ((q >> 1) << 20), __double2loint(x));
}
__device__ __forceinline__ double recip_pos(double v) {
  const int hi = __double2hiint(v), e = hi >> 20;
  if ((unsigned)(e - 1) >= 0x7fcu) return __drcp_rn(v);
  const double m = __hiloint2double(hi - ((e - 1023) << 20), __double2loint(v));
  const double x0 = f64_of_f32_scaled(__fdividef(1.0f, f32_of_normal(m)), 0);
  const double r = fma(-m, x0, 1.0);
  const double x = fma(x0, fma(r, r, r), x0);
  return __hiloint2double(__double2hiint(x) - ((e - 1023) << 20), __double2loint(x));
}

// The rotation of a pair of columns a, b of a one-sided Jacobi SVD: squared
// norms na, nb, dot product g.  Two lanes of a warp may hold a pair with na
// and nb exchanged and have to agree: every expression in na and nb is
// symmetric in FP32, too.

// Smallest |g| that is rotated, 2.5e-15 ||a|| ||b||.
__device__ __forceinline__ float jacobi_threshold(double na, double nb) {
  const float ra = f32_of_normal(na), rb = f32_of_normal(nb);
  return 2.5e-15f * ((ra * rsqrtf(ra)) * (rb * rsqrtf(rb)));
}

// tan(theta), the smaller root of t^2 + 2 z t - 1, z = d / 2 g with d = nb - na:
// sign(z) / (|z| + sqrt(z^2 + 1)); 0: no rotation (|g| <= thr, or not finite).
__device__ __forceinline__ float jacobi_tan(float g, float d, float thr) {
  if (!(fabsf(g) > thr)) return 0.0f;
  const float z = __fdividef(d, 2.0f * g), az = fabsf(z), z2 = fmaf(az, az, 1.0f);
  const float den = az < 1e9f ? az + z2 * rsqrtf(z2) : 2.0f * az;
  const float t = copysignf(__fdividef(1.0f, den), z);
  return fabsf(t) <= 1.0f ? t : 0.0f;
}

// 1 / sqrt(q), q = 1 + t^2, from an FP32 seed c0 by one step of third order,
// c0 (1 + e / 2 + 3 e^2 / 8), e = 1 - q c0^2.
__device__ __forceinline__ double jacobi_cos(double q, float t) {
  const double c0 = f64_of_f32_scaled(rsqrtf(fmaf(t, t, 1.0f)), 0);
  const double e = fma(-(q * c0), c0, 1.0);
  return fma(c0, e * fma(e, 0.375, 0.5), c0);
}

}  // namespace h2
