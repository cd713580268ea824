// Orthonormalising coefficients of a small Gram matrix, one CTA; included by
// small.cu (one matrix per launch) and batch.cu (one CTA per molecule).
#pragma once

#include <cuda_runtime.h>

#include "f64_estimates.cuh"

namespace xs {
namespace {

// smallest eigenvalue of the Gram matrix, relative to its largest diagonal entry and
// to one (the square of the unit rows that Gram-Schmidt started from), that the
// triangular factor serves
constexpr double kOrthPivot = 1e-9;

// B = L^-1 for the n x n Gram matrix G = L L^T in A (row stride ld, overwritten;
// its lower triangle is read), B row stride ld, both in shared memory; false
// (with A and B spoilt) when a pivot falls to kOrthPivot of max(1, largest diagonal
// entry), or when |B|_F^2 = trace(G^-1), which 1 / lambda_min cannot exceed, leaves
// lambda_min below that (pivots without exchanges alone do not bound it: the rows of
// a Kahan matrix).  So every direction that Loewdin's absolute rule (1e-14 of
// max(1, lambda_max), lambda_max <= 64 diagonal entries) would drop goes to Loewdin:
// a block that Gram-Schmidt reduced to rounding noise is not scaled back to unit
// rows.  The rows of B T are then orthonormal, like the Loewdin rows
// Lambda^-1/2 Q^T T but rotated; both are as orthonormal as the rounding of G
// lets them be (2^-53 over its smallest eigenvalue).  Right-looking elimination on
// [G | I]: n steps of about 700 cycles, against eight Jacobi sweeps of n rounds of
// 3000 (20 rows: under 14 us instead of 215).
__device__ bool gram_inverse_factor(int n, double* A, double* B, int ld) {
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int idx = tid; idx < n * n; idx += nt) B[(idx / n) * ld + idx % n] = idx / n == idx % n ? 1.0 : 0.0;
  long long top = 0;
  for (int i = 0; i < n; ++i) top = max(top, __double_as_longlong(A[i * ld + i]));   // non-negative diagonal
  const double least = kOrthPivot * fmax(__longlong_as_double(top), 1.0);
  const float rn = 1.0f / static_cast<float>(n);
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    const double x = A[j * ld + j];
    if (!(mag_bits(x) > mag_bits(least)) || __double2hiint(x) < 0 || __double2hiint(x) >= 0x7FF00000) return false;
    if (tid < ((n + 31) & ~31)) {
      const double r = rsqrt_full(x);
      // column j of L below the pivot, row j of B
      if (tid > j && tid < n) A[tid * ld + j] *= r;
      else if (tid <= j) B[j * ld + tid] *= r;
    }
    __syncthreads();
    const int work = (n - 1 - j) * n;
    for (int q = tid; q < work; q += nt) {
      int g = static_cast<int>((static_cast<float>(q) + 0.5f) * rn);
      if (g * n > q) --g;
      const int i = j + 1 + g, c = q - g * n;
      const double l = A[i * ld + j];
      if (c <= j) B[i * ld + c] = fma(-l, B[j * ld + c], B[i * ld + c]);
      else if (c <= i) A[i * ld + c] = fma(-l, A[c * ld + j], A[i * ld + c]);
    }
    __syncthreads();
  }
  // |B|_F^2 in float32
  __shared__ float part[32];
  float f = 0.0f;
  for (int q = tid; q < n * n; q += nt) {
    const double x = B[(q / n) * ld + q % n];
    const float y = float_range(x) ? narrow_bits(x) : (mag_bits(x) > mag_bits(1.0) ? 1e30f : 0.0f);
    f = fmaf(y, y, f);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
  if ((tid & 31) == 0) part[tid >> 5] = f;
  __syncthreads();
  f = 0.0f;
  for (int w = 0; w < nt >> 5; ++w) f += part[w];
  return f * static_cast<float>(least) <= 1.0f;
}

}  // namespace
}  // namespace xs
