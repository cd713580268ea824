"""One residue product C = A B^T against exact rational arithmetic, on rows whose
entries spread over many decades.

Row a is rounded to integers of 2^-57 of 2^ea, |a| <= 2^ea < 2.01 |a|, so every entry
is off by at most 2^-58 2^ea; the integer product is exact and rounded once:
|C - a.b| <= 2^-58 (2^ea sum|b| + 2^eb sum|a|) (1 + 2^-50) + 2^-53 |C|.  The error is
relative to the rows' norms, not to the products that meet in an output.
"""
import ctypes
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "modgemm.h"
template <typename T> static T* up(const T* h, size_t n) {
  T* d; cudaMalloc(&d, n * sizeof(T)); cudaMemcpy(d, h, n * sizeof(T), cudaMemcpyHostToDevice); return d;
}
// A: M x K (acols: stored K x M), B: N x K (bcols likewise)
extern "C" int product(int M, int N, int K, const double* A, int acols, const double* B, int bcols, double* C) {
  double *a = up(A, (size_t)M * K), *b = up(B, (size_t)N * K), *c;
  const int zero = 0;
  int *err = up(&zero, 1), e = 0;
  cudaMalloc(&c, sizeof(double) * M * N);
  {
    xs::MgPlanes pa, pb;
    xs::MgWork w;
    xs::MgOperand x{a, acols ? 1 : K, acols ? M : 1, 0, M, K, 1}, y{b, bcols ? 1 : K, bcols ? N : 1, 0, N, K, 1};
    xs::mg_split(nullptr, 0, x, pa);
    xs::mg_split(nullptr, 1, y, pb);
    xs::MgOut o;
    o.C = c; o.ldc = N; o.sC = (long long)M * N;
    xs::mg_product(nullptr, x, y, 1, o, w, err);
    cudaMemcpy(C, c, sizeof(double) * M * N, cudaMemcpyDeviceToHost);
    cudaMemcpy(&e, err, sizeof(int), cudaMemcpyDeviceToHost);
  }
  cudaFree(a); cudaFree(b); cudaFree(c); cudaFree(err);
  return e ? e : static_cast<int>(cudaDeviceSynchronize());
}
"""


@pytest.fixture(scope="module")
def product(tmp_path_factory):
    from tests.device_code import compile_and_load
    lib = compile_and_load(str(tmp_path_factory.mktemp("residues")), "residues", SOURCE)

    def call(A, B, acols, bcols):
        C = np.zeros((len(A), len(B)))
        a, b = np.ascontiguousarray(A.T if acols else A), np.ascontiguousarray(B.T if bcols else B)
        p = lambda x: ctypes.c_void_p(x.ctypes.data)
        assert lib.product(len(A), len(B), A.shape[1], p(a), int(acols), p(b), int(bcols), p(C)) == 0
        return C
    return call


def _graded(rng, rows, K, decades):
    """Entries over `decades` decades, rows scaled by 2^-300 to 2^300, a zero row."""
    x = rng.standard_normal((rows, K)) * 10.0 ** rng.uniform(-decades, 0.0, (rows, K))
    x[:, rng.integers(0, K, 2)] = 0.0
    x[0] = 0.0
    return np.ldexp(x, rng.integers(-300, 301, (rows, 1)))


def _exponent(row):
    """ea of the row (the norm from float64, well inside the 2^-9 by which it is overestimated)."""
    m = np.abs(row).max()
    if m == 0.0:
        return 0
    e = int(np.floor(np.log2(m)))
    n = np.linalg.norm(np.ldexp(row, -e))
    return e + int(np.ceil(np.log2(n * 1.001)))


@pytest.mark.parametrize("K", [1, 63, 64, 300, 1025])
@pytest.mark.parametrize("decades", [0, 20, 60])
@pytest.mark.parametrize("acols,bcols", [(False, False), (True, True)])
def test_graded_rows(product, K, decades, acols, bcols):
    rng = np.random.default_rng(K + decades)
    A, B = _graded(rng, 5, K, decades), _graded(rng, 4, K, decades)
    # large entries that meet only small ones: |a.b| far below |a| |b|
    if K > 2:
        A[1, : K // 2] *= 1e-12
        B[1, K // 2:] *= 1e-12
    C = product(A, B, acols, bcols)
    fa, fb = [[Fraction(float(v)) for v in r] for r in A], [[Fraction(float(v)) for v in r] for r in B]
    for i in range(len(A)):
        for j in range(len(B)):
            exact = sum(x * y for x, y in zip(fa[i], fb[j]))
            ea, eb = Fraction(2) ** _exponent(A[i]), Fraction(2) ** _exponent(B[j])
            bound = (ea * sum(map(abs, fb[j])) + eb * sum(map(abs, fa[i]))) * Fraction(2) ** -58 * (1 + Fraction(2) ** -50)
            assert abs(Fraction(float(C[i, j])) - exact) <= bound + abs(exact) * Fraction(2) ** -53
