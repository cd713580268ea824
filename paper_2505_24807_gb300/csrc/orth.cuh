// Orthonormalising coefficients of a small Gram matrix, one CTA; included by
// small.cu (one matrix per launch) and batch.cu (one CTA per molecule).
#pragma once

#include <cuda_runtime.h>

#include "f64_estimates.cuh"

namespace xs {
namespace {

// smallest Cholesky pivot, relative to the largest diagonal entry, that the
// triangular factor serves
constexpr double kOrthPivot = 1e-9;

// B = L^-1 for the n x n Gram matrix G = L L^T in A (row stride ld, overwritten;
// its lower triangle is read), B row stride ld, both in shared memory; false
// (with A and B spoilt) when a pivot falls to kOrthPivot of the largest diagonal
// entry.  The rows of B T are then orthonormal, like the Loewdin rows
// Lambda^-1/2 Q^T T but rotated; both are as orthonormal as the rounding of G
// lets them be (2^-53 over its smallest eigenvalue), and above kOrthPivot the
// Loewdin factors drop no direction.  Right-looking elimination on [G | I]: n
// steps of about 700 cycles, against eight Jacobi sweeps of n rounds of 3000
// (20 rows: under 14 us instead of 215).
__device__ bool gram_inverse_factor(int n, double* A, double* B, int ld) {
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int idx = tid; idx < n * n; idx += nt) B[(idx / n) * ld + idx % n] = idx / n == idx % n ? 1.0 : 0.0;
  long long top = 0;
  for (int i = 0; i < n; ++i) top = max(top, __double_as_longlong(A[i * ld + i]));   // non-negative diagonal
  const double least = kOrthPivot * __longlong_as_double(top);
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
  return true;
}

}  // namespace
}  // namespace xs
