"""Rayleigh-Ritz eigensolver on the matrices of a restarted Davidson solve: the Ritz
values on the diagonal and a few new rows whose couplings to them run from the size of
an unconverged root's residual down to rounding, and wholly diagonal ones.

Backward stability as in test_gpu_eig_sizes.py: 20 S^2 2^-53 |A| / S for a spectrum of
norm |A| and gaps of at least |A| / S.
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


def _restarted(S, new, decades, seed):
    """Eigenvalues near 1 .. S with a random fraction, so that they round to float32."""
    rng = np.random.default_rng(seed)
    A = np.diag(np.arange(1.0, S + 1.0) + 0.2 * rng.random(S))
    c = rng.standard_normal((new, S - new)) * 10.0 ** rng.uniform(-decades, -4.0, (new, S - new))
    A[S - new:, : S - new] = c
    A[: S - new, S - new:] = c.T
    return A


@pytest.mark.parametrize("S,k,new", [(3, 2, 1), (28, 26, 2), (40, 32, 1), (96, 64, 8), (150, 20, 3), (230, 40, 2)])
@pytest.mark.parametrize("decades", [6, 14, 30, 200])
def test_restarted_subspaces(ctx, S, k, new, decades):
    bound = 20.0 * max(S, 4) ** 2 * 2.0 ** -53
    for seed in range(20):
        A = _restarted(S, new, decades, 100 * S + seed)
        w, Z = xs.xs_subspace_eig(ctx.h, A, k)
        assert np.abs(w - np.linalg.eigvalsh(A)[:k]).max() < bound
        assert np.abs(A @ Z - Z * w).max() < bound
        assert np.abs(Z.T @ Z - np.eye(k)).max() < bound


@pytest.mark.parametrize("S,k", [(1, 1), (20, 20), (130, 40)])
def test_diagonal(ctx, S, k):
    for seed in range(10):
        d = np.random.default_rng(seed).permutation(np.arange(1.0, S + 1.0) + 0.2 * np.random.default_rng(seed).random(S))
        w, Z = xs.xs_subspace_eig(ctx.h, np.diag(d), k)
        assert np.abs(w - np.sort(d)[:k]).max() < 20.0 * S ** 2 * 2.0 ** -53
        assert np.abs(Z.T @ Z - np.eye(k)).max() < 20.0 * max(S, 4) ** 2 * 2.0 ** -53
