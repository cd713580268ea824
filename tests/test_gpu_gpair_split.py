"""The float32 G build deals its vectors out to CTAs: numbers of vectors that leave a
last, shorter share, on TF32 pairs (501 AOs) and on float16 pairs (1233 AOs), against the float64
products within the mixed products' bound."""
import numpy as np
import pytest

import molgen
from tests.gpu_common import context, mixed_product_err, mixed_product_tol

pytestmark = pytest.mark.gpu

xs = pytest.importorskip("paper_2505_24807_gb300.xs")


@pytest.mark.parametrize("heavy,h,nvec", [(85, 161, 70), (233, 301, 13)])
def test_vector_shares(heavy, h, nvec):
    ctx = context(molgen.make_params(0))
    try:
        xs.xs_ground_state(ctx.h, [molgen.make_chain(3, heavy, h)], scf_tol=1e-3)
        n, o, _ = xs.xs_get_sizes(ctx.h, 0)
        assert n == 4 * heavy + h
        _, eps = xs.xs_get_orbitals(ctx.h, 0)
        X = molgen.trial_vectors(5, nvec, o, n - o).reshape(nvec, -1) / np.sqrt(o * (n - o))
        for kind in (xs.XS_KIND_A, xs.XS_KIND_APB, xs.XS_KIND_AMB):
            ref = xs.xs_apply(ctx.h, 0, kind, X)
            Y = xs.xs_apply(ctx.h, 0, kind, X, precision=1)
            assert mixed_product_err(Y, ref, X, eps, o) < mixed_product_tol(n)
    finally:
        ctx.close()
