"""Float64 products whose transforms run as residue products on the tensor cores.

The residue products carry 57-bit integers and round once, so each of the four
chained products of A X is at least as accurate as a float64 GEMM; the oracle's
own GEMMs bound the difference by about n 2^-53 relative per product: 1e-12 of
the largest entry covers four of them and the two-electron sums at n <= 250.
"""
import numpy as np
import pytest

import molgen
from tests.gpu_common import context, oracle_ground_state, rel_err

pytestmark = pytest.mark.gpu

xs = pytest.importorskip("paper_2505_24807_gb300.xs")


# heavy atoms, hydrogens, vectors: AO counts around the rule's lines (96 and 160
# AOs, small batches), nocc == nvir and nvir < nocc, K and N off the tile sizes
@pytest.mark.parametrize("heavy,h,nvec", [(18, 24, 20), (30, 41, 1), (31, 45, 3), (40, 82, 2), (45, 70, 9)])
def test_residue_products_match_oracle(heavy, h, nvec):
    from oracle import excited
    params = molgen.make_params(0)
    Z, xyz = molgen.make_chain(3, heavy, h)
    mol, ints, res = oracle_ground_state(Z, xyz, params)
    ctx = context(params)
    try:
        xs.xs_ground_state(ctx.h, [(Z, xyz)], scf_tol=1e6)
        xs.xs_set_orbitals(ctx.h, 0, res.C, res.eps)
        X = molgen.trial_vectors(5, nvec, mol.nocc, mol.nvir)
        for kind, okind in ((0, "A"), (1, "ApB"), (2, "AmB")):
            Y = xs.xs_apply(ctx.h, 0, kind, X.reshape(nvec, -1)).reshape(X.shape)
            ref = excited.apply_kind(mol, ints, res.C, res.eps, mol.nocc, X, okind)
            assert rel_err(Y, ref) < 1e-12
    finally:
        ctx.close()


def test_residue_products_special_inputs():
    """Non-finite entries stay in their own vector, zero vectors give zero, and a
    power of two on a vector comes out as that power of two on its product."""
    params = molgen.make_params(0)
    Z, xyz = molgen.make_chain(3, 40, 62)
    ctx = context(params)
    try:
        xs.xs_ground_state(ctx.h, [(Z, xyz)])
        n, o, _ = xs.xs_get_sizes(ctx.h, 0)
        X = molgen.trial_vectors(5, 5, o, n - o).reshape(5, -1)
        Y = xs.xs_apply(ctx.h, 0, 0, X)
        X2 = X.copy()
        X2[1, 77] = np.nan
        X2[2, 5] = np.inf
        X2[3] = 0.0
        X2[4] *= 2.0 ** -600
        Y2 = xs.xs_apply(ctx.h, 0, 0, X2)
        assert np.array_equal(Y2[0], Y[0])
        assert np.isnan(Y2[1]).all()
        assert not np.isfinite(Y2[2]).any()
        assert not Y2[3].any()
        assert np.array_equal(Y2[4], Y[4] * 2.0 ** -600)
    finally:
        ctx.close()


def test_residue_products_in_chunks():
    """A batch beyond the residue planes' budget runs in chunks: each vector's
    product is the one it has alone (the two-electron sums may group differently)."""
    params = molgen.make_params(0)
    Z, xyz = molgen.make_chain(3, 170, 300)
    ctx = context(params)
    try:
        xs.xs_ground_state(ctx.h, [(Z, xyz)], scf_tol=1e6)
        n, o, _ = xs.xs_get_sizes(ctx.h, 0)
        X = molgen.trial_vectors(5, 27, o, n - o).reshape(27, -1)
        Y = xs.xs_apply(ctx.h, 0, 1, X)
        for k in (0, 21, 22, 26):
            one = xs.xs_apply(ctx.h, 0, 1, X[k:k + 1])
            assert rel_err(Y[k:k + 1], one) < 1e-13
    finally:
        ctx.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_device_arrays_in_place(precision):
    """Products on device arrays are used in place: aligned, misaligned (8 bytes),
    overlapping and identical input and output give the host arrays' result."""
    torch = pytest.importorskip("torch")
    params = molgen.make_params(0)
    Z, xyz = molgen.make_chain(3, 30, 41)
    ctx = context(params)
    try:
        xs.xs_ground_state(ctx.h, [(Z, xyz)], scf_tol=1e6)
        n, o, _ = xs.xs_get_sizes(ctx.h, 0)
        ov = o * (n - o)
        X = molgen.trial_vectors(5, 3, o, n - o).reshape(3, -1)
        ref = xs.xs_apply(ctx.h, 0, 1, X, precision=precision)
        buf = torch.zeros(8 * ov + 8, dtype=torch.float64, device="cuda")
        for at_in, at_out in ((0, 4 * ov), (1, 4 * ov + 1), (0, ov), (2 * ov, 0), (0, 0)):
            x, y = buf[at_in:at_in + 3 * ov].view(3, ov), buf[at_out:at_out + 3 * ov].view(3, ov)
            x.copy_(torch.from_numpy(X))
            torch.cuda.synchronize()
            xs.xs_apply(ctx.h, 0, 1, x, precision=precision, out=y)
            assert np.array_equal(y.cpu().numpy(), ref)
        A = torch.randn(5, 1001, dtype=torch.float64, device="cuda")
        B = torch.randn(3, 1001, dtype=torch.float64, device="cuda")
        out = torch.empty(5, 3, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        xs._check(ctx.h, xs.load().xs_subspace_gram(ctx.h, 5, 3, 1001, xs._ptr(A), xs._ptr(B), xs._ptr(out), 1))
        assert np.array_equal(out.cpu().numpy(), xs.xs_subspace_gram(ctx.h, A.cpu().numpy(), B.cpu().numpy()))
        # the output on top of the input
        Xs, c = torch.randn(1, 5, 1001, dtype=torch.float64, device="cuda"), np.random.default_rng(1).standard_normal((1, 5, 3))
        ref = xs.xs_subspace_combine(ctx.h, Xs.cpu().numpy(), c)
        xs._check(ctx.h, xs.load().xs_subspace_combine(ctx.h, 1, 5, 3, 1001, xs._ptr(Xs), xs._ptr(c), xs._ptr(Xs), 1))
        assert np.array_equal(Xs[0, :3].cpu().numpy(), ref)
    finally:
        ctx.close()
