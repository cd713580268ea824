"""Rayleigh-Ritz eigensolver on degenerate eigenvalues with others close by (identical
fragments: pairs that differ from each other by 1e-6 to 1e-3 of |A|).

Residuals to a backward error of 20 S 2^-53 |A|; vectors orthonormal to 1e-9, the bound
of test_gpu_subspace.py.
"""
import numpy as np
import pytest

import molgen
from tests.gpu_common import context

pytestmark = pytest.mark.gpu

xs = pytest.importorskip("paper_2505_24807_gb300.xs")

PATTERNS = {   # eigenvalues in units of the gap, above 10
    "pair, pair": [0, 0, 1, 1],
    "pair, one": [0, 0, 1],
    "one, pair": [0, 1, 1],
    "four, one": [0, 0, 0, 0, 1],
    "three pairs": [0, 0, 1, 1, 2.5, 2.5],
    "six, pair": [0, 0, 0, 0, 0, 0, 1, 1],
}


@pytest.fixture(scope="module")
def ctx():
    c = context(molgen.make_params(0))
    yield c
    c.close()


@pytest.mark.parametrize("pattern", sorted(PATTERNS))
@pytest.mark.parametrize("gap", [2.2e-6, 4e-6, 7e-6, 1e-5, 1.2e-5, 3e-5, 1e-4, 1e-3])
def test_close_clusters(ctx, pattern, gap):
    rng = np.random.default_rng(int(1e7 * gap))
    for _ in range(8):
        S = int(rng.integers(20, 100))
        lam = np.r_[10.0 + rng.random() * 1e-3 + 20.0 * gap * np.array(PATTERNS[pattern]), rng.uniform(10.5, 20.0, S - 10)]
        S = len(lam)
        q, _ = np.linalg.qr(rng.standard_normal((S, S)))
        A = (q * lam) @ q.T
        A = 0.5 * (A + A.T)
        k = min(S, 12)
        w, Z = xs.xs_subspace_eig(ctx.h, A, k)
        bound = 20.0 * S * 2.0 ** -53 * 20.0
        assert np.abs(w - np.sort(lam)[:k]).max() < bound
        assert np.abs(A @ Z - Z * w).max() < bound
        assert np.abs(Z.T @ Z - np.eye(k)).max() < 1e-9
