"""Orthonormalising coefficients of one Gram matrix: how many directions are kept
(Loewdin's rule: eigenvalues above 1e-14 max(1, lambda_max)) and how orthonormal
they come out, where the triangular factor could mistake dependent rows for
independent ones.

G is rounded to n 2^-53 lambda_max, and a kept direction is scaled by
1 / sqrt(lambda): |Q Q^T - I| is at most 4 n 2^-53 lambda_max / (least kept lambda).
"""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

THRESH = 1e-14

SOURCE = r"""
#include "small.h"
extern "C" int orth(int n, const double* G, double* B, int* nkeep) {
  double *g, *v, *w, *b;
  int* k;
  const size_t nn = sizeof(double) * n * n;
  cudaMalloc(&g, nn); cudaMalloc(&v, nn); cudaMalloc(&w, sizeof(double) * n); cudaMalloc(&b, nn); cudaMalloc(&k, 2 * sizeof(int));
  cudaMemcpy(g, G, nn, cudaMemcpyHostToDevice);
  xs::orthonormaliser(nullptr, n, g, n, v, n, w, 1e-14, b, n, k, k + 1);
  cudaMemcpy(B, b, nn, cudaMemcpyDeviceToHost);
  cudaMemcpy(nkeep, k, sizeof(int), cudaMemcpyDeviceToHost);
  cudaFree(g); cudaFree(v); cudaFree(w); cudaFree(b); cudaFree(k);
  return static_cast<int>(cudaDeviceSynchronize());
}
"""


@pytest.fixture(scope="module")
def orth(tmp_path_factory):
    from tests.device_code import compile_and_load
    lib = compile_and_load(str(tmp_path_factory.mktemp("orth")), "orth", SOURCE)

    def call(G):
        n = len(G)
        G = np.ascontiguousarray(G)
        B = np.zeros((n, n))
        k = ctypes.c_int(-1)
        assert lib.orth(n, ctypes.c_void_p(G.ctypes.data), ctypes.c_void_p(B.ctypes.data), ctypes.byref(k)) == 0
        return B[:k.value], k.value
    return call


def _rows(n, scale, seed):
    """n rows of norm `scale`, well apart."""
    rng = np.random.default_rng(seed)
    return scale * (np.eye(n, n + 3) + 0.2 * rng.standard_normal((n, n + 3)) / np.sqrt(n))


@pytest.mark.parametrize("n", [1, 2, 20, 33, 64])
@pytest.mark.parametrize("norm", [1.0, 1e-3, 1e-6, 1e-8, 1e-15])
def test_small_rows(orth, n, norm):
    """A whole block that Gram-Schmidt left with norm `norm`: kept or dropped by the
    absolute rule."""
    T = _rows(n, norm, n)
    ev = np.linalg.eigvalsh(T @ T.T)
    keep = int((ev > THRESH * max(1.0, ev[-1])).sum())
    assert keep in (0, n)
    B, k = orth(T @ T.T)
    assert k == keep
    if k:
        Q = B @ T
        assert np.abs(Q @ Q.T - np.eye(k)).max() < 4 * n * 2.0 ** -53 * ev[-1] / ev[0]


@pytest.mark.parametrize("n,s", [(20, 0.7), (32, 0.75), (64, 0.87)])
def test_graded_rows(orth, n, s):
    """Rows of a Kahan matrix: unit norms and elimination pivots above 1e-8 with one
    direction that is dependent to rounding."""
    R = (s ** np.arange(n))[:, None] * (np.eye(n) - np.triu(np.full((n, n), np.sqrt(1.0 - s * s)), 1))
    T = np.ascontiguousarray(R.T)
    ev = np.linalg.eigvalsh(T @ T.T)
    assert abs(ev[0]) < THRESH * ev[-1] < 1e-3 * ev[1]
    B, k = orth(T @ T.T)
    assert k == n - 1
    Q = B @ T
    assert np.abs(Q @ Q.T - np.eye(k)).max() < 4 * n * 2.0 ** -53 * ev[-1] / ev[1]
