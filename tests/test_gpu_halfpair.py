"""Mixed products on float16 pairs (molecules of at least 512 AOs) against the
float64 products, within the bound of the mixed products' four split GEMMs
(mixed_product_tol: the pairs' two 11-bit significands are those of a TF32 pair,
and half as many accumulation steps truncate)."""
import numpy as np
import pytest

import molgen
from tests.gpu_common import context, mixed_product_err, mixed_product_tol

pytestmark = pytest.mark.gpu

xs = pytest.importorskip("paper_2505_24807_gb300.xs")


def _load(heavy, h):
    ctx = context(molgen.make_params(0))
    xs.xs_ground_state(ctx.h, [molgen.make_chain(3, heavy, h)], scf_tol=1e-4)
    n, o, _ = xs.xs_get_sizes(ctx.h, 0)
    _, eps = xs.xs_get_orbitals(ctx.h, 0)
    return ctx, n, o, eps


# nocc == nvir (the alkane) and nvir < nocc, row lengths that allow 16-byte
# accesses and odd ones, one vector, a batch past a group of 8
@pytest.mark.parametrize("heavy,h,nvec", [(86, 174, 2), (87, 165, 1), (90, 161, 9), (97, 190, 3)])
def test_half_pair_products(heavy, h, nvec):
    ctx, n, o, eps = _load(heavy, h)
    try:
        assert n >= 512
        X = molgen.trial_vectors(5, nvec, o, n - o).reshape(nvec, -1) / np.sqrt(o * (n - o))
        for kind in (xs.XS_KIND_A, xs.XS_KIND_APB, xs.XS_KIND_AMB, xs.XS_KIND_A_TRIPLET, xs.XS_KIND_APB_TRIPLET):
            ref = xs.xs_apply(ctx.h, 0, kind, X)
            Y = xs.xs_apply(ctx.h, 0, kind, X, precision=1)
            assert mixed_product_err(Y, ref, X, eps, o) < mixed_product_tol(n)
    finally:
        ctx.close()


def test_half_pair_special_inputs():
    """Powers of two pass through exactly (within float32's range), also when one
    entry dominates a vector; zero vectors give zero; non-finite entries stay in
    their own vector."""
    ctx, n, o, eps = _load(87, 165)
    try:
        X = molgen.trial_vectors(5, 6, o, n - o).reshape(6, -1) / np.sqrt(o * (n - o))
        X[3] *= 1e-3
        X[3, 11] = 1.0
        ref = xs.xs_apply(ctx.h, 0, xs.XS_KIND_APB, X, precision=1)
        full = xs.xs_apply(ctx.h, 0, xs.XS_KIND_APB, X)
        assert mixed_product_err(ref, full, X, eps, o) < mixed_product_tol(n)
        X2 = X.copy()
        X2[0] *= 2.0 ** 60
        X2[1] *= 2.0 ** -60
        X2[2] = 0.0
        X2[4, 5] = np.inf
        X2[5, 7] = np.nan
        Y = xs.xs_apply(ctx.h, 0, xs.XS_KIND_APB, X2, precision=1)
        assert np.array_equal(Y[0], ref[0] * 2.0 ** 60)
        assert np.array_equal(Y[1], ref[1] * 2.0 ** -60)
        assert not Y[2].any()
        assert np.array_equal(Y[3], ref[3])
        assert not np.isfinite(Y[4:]).all(axis=1).any()
    finally:
        ctx.close()
