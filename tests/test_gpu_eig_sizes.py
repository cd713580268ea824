"""Rayleigh-Ritz eigensolver at the sizes where its blocks end.

A = Q diag(1, .., S) Q^T has gaps of 1 and norm S, so a backward error of a few
S 2^-53 |A| moves eigenvalues by that and eigenvectors by that over the gap:
bounds of 20 S^2 2^-53 for residuals and for the deviation from orthonormality.
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


# one warp and two, the reflector blocks of 8, the shared-memory limits of the
# scratch (6 S k) and of the matrix (224), one row past it
@pytest.mark.parametrize("S,k", [(1, 1), (2, 1), (3, 3), (8, 8), (10, 4), (11, 11), (32, 5), (33, 33), (34, 1), (64, 20),
                                 (65, 10), (97, 40), (129, 12), (160, 20), (223, 7), (224, 10), (225, 10), (300, 33)])
def test_eigensolver_sizes(ctx, S, k):
    q = molgen.orthonormal_matrix(S, S)
    A = (q * np.arange(1.0, S + 1.0)) @ q.T
    A = 0.5 * (A + A.T)
    w, Z = xs.xs_subspace_eig(ctx.h, A, k)
    bound = 20.0 * max(S, 4) ** 2 * 2.0 ** -53
    assert np.abs(w - np.arange(1.0, k + 1.0)).max() < bound
    assert np.abs(A @ Z - Z * w).max() < bound
    assert np.abs(Z.T @ Z - np.eye(k)).max() < bound


def test_eigensolver_scales_and_zero_columns(ctx):
    """Already tridiagonal and diagonal matrices (reflectors that are the identity)
    and entries far from one (beyond the float32 range of the estimates)."""
    S, k = 40, 6
    T = np.diag(np.arange(1.0, S + 1.0)) + np.diag(np.full(S - 1, 0.25), 1) + np.diag(np.full(S - 1, 0.25), -1)
    bound = 20.0 * S ** 2 * 2.0 ** -53
    for A, scale in ((T, 1.0), (np.diag(np.arange(1.0, S + 1.0)), 1.0), (T * 2.0 ** 30, 2.0 ** 30),
                     (T * 2.0 ** -30, 2.0 ** -30)):
        w, Z = xs.xs_subspace_eig(ctx.h, A, k)
        ref = np.linalg.eigvalsh(A)[:k]
        assert np.abs(w - ref).max() < bound * scale
        assert np.abs(A @ Z - Z * w).max() < bound * scale
        assert np.abs(Z.T @ Z - np.eye(k)).max() < bound
