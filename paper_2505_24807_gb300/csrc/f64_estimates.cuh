// Float64 reciprocals and roots of libxs's small dense kernels from float32
// estimates.  A float64 instruction of a warp holds its sub-partition's pipe for
// 64 cycles on this part; the library's square root takes 610 cycles, its
// division and reciprocal square root 380 (one warp, measured), these 250 to 320.
#pragma once

#include <cuda_runtime.h>

namespace xs {
namespace {

// |x| as an integer that orders like it: comparisons stay off the float64 pipe
__device__ __forceinline__ long long mag_bits(double x) { return __double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFll; }

// float32 of a double and back by their fields (the conversion instructions run
// on the float64 pipe, 64 cycles each), for 2^-120 < |x| < 2^120
__device__ __forceinline__ bool float_range(double x) {
  const int e = (__double2hiint(x) >> 20) & 0x7FF;
  return e > 1023 - 120 && e < 1023 + 120;
}
__device__ __forceinline__ float narrow_bits(double x) {
  const unsigned hi = static_cast<unsigned>(__double2hiint(x)), lo = static_cast<unsigned>(__double2loint(x));
  return __uint_as_float((hi & 0x80000000u) | (((hi & 0x7FFFFFFFu) - (896u << 20)) << 3) | (lo >> 29));
}
__device__ __forceinline__ double widen_bits(float x) {
  const unsigned u = __float_as_uint(x);
  return __hiloint2double(static_cast<int>((u & 0x80000000u) | (((u & 0x7FFFFFFFu) >> 3) + (896u << 20))),
                          static_cast<int>(u << 29));
}
__device__ __forceinline__ float rcp_estimate(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float rsqrt_estimate(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// The corrections are binomial series (Householder's iterations of the first and second
// order) in the residual e of a float32 estimate r, |e| <= 2^-19:
//   1 / x = r / (1 - e),           e = 1 - x r:     r (1 + e + e^2 + ...)
//   1 / sqrt(x) = r (1 - e)^-1/2,  e = 1 - x r^2:   r (1 + e / 2 + 3 e^2 / 8 + ...)
//   sqrt(x) = x r (1 - e)^-1/2

// reciprocal to 2^-45 relative (seen), the first order (inverse iteration needs
// directions, not correctly rounded quotients)
__device__ __forceinline__ double rcp_fast(double x) {
  if (!float_range(x)) return 1.0 / x;
  const double r = widen_bits(rcp_estimate(narrow_bits(x)));
  return r * fma(-x, r, 2.0);
}

// square root, its reciprocal and the reciprocal (x > 0 for the roots), the second
// order: the terms left out are e^3 (below 2^-57), 2 ulp with the roundings (1 seen)
__device__ __forceinline__ double sqrt_fast(double x) {
  if (!float_range(x)) return sqrt(x);
  const double r = widen_bits(rsqrt_estimate(narrow_bits(x)));
  const double t = x * r;
  const double e = fma(-t, r, 1.0);
  return fma(t, e * fma(0.375, e, 0.5), t);
}
__device__ __forceinline__ double rsqrt_full(double x) {
  if (!float_range(x)) return 1.0 / sqrt(x);
  const double r = widen_bits(rsqrt_estimate(narrow_bits(x)));
  const double e = fma(-(x * r), r, 1.0);
  return fma(r, e * fma(0.375, e, 0.5), r);
}
__device__ __forceinline__ double rcp_full(double x) {
  if (!float_range(x)) return 1.0 / x;
  const double r = widen_bits(rcp_estimate(narrow_bits(x)));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

}  // namespace
}  // namespace xs
