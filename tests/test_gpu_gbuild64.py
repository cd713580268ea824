"""Float64 G build (Coulomb partial sums, tiles and their mirrored blocks) at its
edges: column tiles of 64 AOs cut by atoms, hydrogen runs that do not fill a row
group, batches of 1, 8 and 11 vectors (groups of 8 and a remainder), W rows in one
and several partial sums, singlets and triplets.  Both sides are float64 sums of
the same terms: 1e-12 of the largest entry, as for the other products.
"""
import numpy as np
import pytest

import molgen
from tests.gpu_common import context, oracle_ground_state, rel_err

pytestmark = pytest.mark.gpu

xs = pytest.importorskip("paper_2505_24807_gb300.xs")


@pytest.mark.parametrize("heavy,h,nvec", [(1, 4, 1), (6, 9, 8), (17, 26, 11), (52, 79, 3)])
def test_float64_products_all_kinds(heavy, h, nvec):
    from oracle import scf
    params = molgen.make_params(0)
    Z, xyz = molgen.make_chain(3, heavy, h)
    mol, ints, res = oracle_ground_state(Z, xyz, params)
    o = mol.nocc
    Co, Cv = res.C[:, :o], res.C[:, o:]
    X = molgen.trial_vectors(5, nvec, o, mol.nvir)
    jk = [scf.coulomb_exchange(mol, ints, Co @ x @ Cv.T) for x in X]
    G = {xs.XS_KIND_A: lambda J, K: 2 * J - K, xs.XS_KIND_APB: lambda J, K: 4 * J - K - K.T,
         xs.XS_KIND_AMB: lambda J, K: K.T - K, xs.XS_KIND_A_TRIPLET: lambda J, K: -K,
         xs.XS_KIND_APB_TRIPLET: lambda J, K: -K - K.T}
    ctx = context(params)
    try:
        xs.xs_ground_state(ctx.h, [(Z, xyz)], scf_tol=1e6)
        xs.xs_set_orbitals(ctx.h, 0, res.C, res.eps)
        for kind, g in G.items():
            ref = np.array([(res.eps[None, o:] - res.eps[:o, None]) * x + Co.T @ g(J, K) @ Cv
                            for x, (J, K) in zip(X, jk)])
            Y = xs.xs_apply(ctx.h, 0, kind, X.reshape(nvec, -1)).reshape(X.shape)
            assert rel_err(Y, ref) < 1e-12
        R = np.random.default_rng(2).uniform(-1, 1, (nvec, mol.nao, mol.nao))
        ref = np.array([2 * J - K for J, K in (scf.coulomb_exchange(mol, ints, r) for r in R)])
        assert rel_err(xs.xs_apply(ctx.h, 0, xs.XS_KIND_G, R), ref) < 1e-12
    finally:
        ctx.close()
