"""Float64 roots and reciprocals of the small dense kernels against correctly rounded
ones (CUDA's sqrt and division; the reciprocal root from 100-digit arithmetic).

The float32 estimate r of 1/x or 1/sqrt(x) has a relative error d of at most 2^-20 (an
approximate instruction of better than 2^-22 on the leading 24 bits of x).  With
e = 1 - x r (at most 2^-20) or e = 1 - x r^2 (at most 2^-19) the corrections are the
binomial series of 1/(1 - e) up to e^2 and of (1 - e)^-1/2 up to e^2: the first terms
left out are e^3 <= 2^-60 and (5/16) e^3 <= 2^-58, a small part of an ulp (2^-53 to
2^-52).  Rounding: half an ulp of the final fma, and for the roots half the rounding of
x r, which e takes in with the opposite sign.  Below 2 ulp in all.  rcp_fast stops at e:
e^2 <= 2^-40.
"""
import ctypes
from decimal import Decimal, localcontext

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "f64_estimates.cuh"
__global__ void all(int n, const double* x, double* y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  y[i] = xs::sqrt_fast(fabs(x[i]));
  y[n + i] = xs::rsqrt_full(fabs(x[i]));
  y[2 * n + i] = xs::rcp_full(x[i]);
  y[3 * n + i] = xs::rcp_fast(x[i]);
  y[4 * n + i] = sqrt(fabs(x[i]));
  y[5 * n + i] = 1.0 / x[i];
}
extern "C" int estimates(int n, const double* x, double* y) {
  double *dx, *dy;
  cudaMalloc(&dx, sizeof(double) * n);
  cudaMalloc(&dy, sizeof(double) * 6 * n);
  cudaMemcpy(dx, x, sizeof(double) * n, cudaMemcpyHostToDevice);
  all<<<(n + 255) / 256, 256>>>(n, dx, dy);
  cudaMemcpy(y, dy, sizeof(double) * 6 * n, cudaMemcpyDeviceToHost);
  cudaFree(dx);
  cudaFree(dy);
  return static_cast<int>(cudaDeviceSynchronize());
}
"""


@pytest.fixture(scope="module")
def estimates(tmp_path_factory):
    from tests.device_code import compile_and_load
    lib = compile_and_load(str(tmp_path_factory.mktemp("estimates")), "estimates", SOURCE)

    def call(x):
        x, y = np.ascontiguousarray(x), np.zeros((6, len(x)))
        assert lib.estimates(len(x), ctypes.c_void_p(x.ctypes.data), ctypes.c_void_p(y.ctypes.data)) == 0
        return y
    return call


def _ulps(y, ref):
    return np.abs(y - ref) / np.spacing(np.abs(ref))


def _samples(lo, hi, n):
    """Random signs, exponents in [lo, hi) and mantissas; the ends of a binade."""
    rng = np.random.default_rng(abs(hi))
    m = 1.0 + rng.random(n)
    m[: n // 8] = 1.0
    m[n // 8: n // 4] = 2.0 - 2.0 ** -52
    m[n // 4: n // 4 + n // 16] = 1.0 + 2.0 ** -52
    return np.ldexp(m, rng.integers(lo, hi, n)) * rng.choice([-1.0, 1.0], n)


# the estimates' range of 2^+-120, its ends on either side, the range of CUDA's functions
@pytest.mark.parametrize("lo,hi", [(-2, 3), (-119, 120), (-121, -118), (118, 122), (-1000, -121), (121, 1000)])
def test_roots_and_reciprocals(estimates, lo, hi):
    x = _samples(lo, hi, 20000)
    sq, rs, rc, rf, ref_sq, ref_rc = estimates(x)
    assert _ulps(sq, ref_sq).max() <= 2.0
    assert _ulps(rc, ref_rc).max() <= 2.0
    assert (np.abs(rf - ref_rc) / np.abs(ref_rc)).max() <= 2.0 ** -39
    with localcontext() as c:
        c.prec = 100
        exact = np.array([float(1 / Decimal(float(v)).copy_abs().sqrt()) for v in x[:4000]])
    assert _ulps(rs[:4000], exact).max() <= 2.0
