"""Rayleigh-Ritz eigensolver on matrices far from one in size, down to zero.

Its float32 stages square and invert numbers of the matrix's size; the matrix is
brought near one by a power of two first, so the errors relative to that power are
those of an ordinary matrix: a spectrum 1 .. S, gaps of 1 and norm S, hence the
20 S^2 2^-53 of a few S 2^-53 |A| of backward error.
"""
import numpy as np
import pytest

import molgen
from tests.gpu_common import context

pytestmark = pytest.mark.gpu

xs = pytest.importorskip("paper_2505_24807_gb300.xs")


@pytest.fixture(scope="module")
def ctx():
    c = context(molgen.make_params(0))
    yield c
    c.close()


# one entry, one warp, shared memory, global memory; the line of the scaling (2^12),
# float32's range and beyond, either way
@pytest.mark.parametrize("S,k", [(1, 1), (20, 5), (60, 12), (230, 9)])
@pytest.mark.parametrize("power", [-1000, -600, -200, -130, -60, -40, -29, -13, -12, 5, 6, 13, 40, 60, 64, 100, 130, 300, 1000])
def test_eigensolver_scales(ctx, S, k, power):
    q = molgen.orthonormal_matrix(S, S)
    A = (q * np.arange(1.0, S + 1.0)) @ q.T
    A = 0.5 * (A + A.T)
    w, Z = xs.xs_subspace_eig(ctx.h, np.ldexp(A, power), k)
    w = np.ldexp(w, -power)
    bound = 20.0 * max(S, 4) ** 2 * 2.0 ** -53
    assert np.abs(w - np.arange(1.0, k + 1.0)).max() < bound
    assert np.abs(A @ Z - Z * w).max() < bound
    assert np.abs(Z.T @ Z - np.eye(k)).max() < bound


@pytest.mark.parametrize("S,k", [(1, 1), (2, 1), (7, 1), (40, 3)])
def test_eigensolver_zero_matrix(ctx, S, k):
    w, Z = xs.xs_subspace_eig(ctx.h, np.zeros((S, S)), k)
    assert np.array_equal(w, np.zeros(k)) or np.abs(w).max() < 1e-25
    assert np.abs(Z.T @ Z - np.eye(k)).max() < 20.0 * max(S, 4) ** 2 * 2.0 ** -53
