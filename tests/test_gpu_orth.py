"""Block orthonormalisation of the Davidson step at its sizes: new blocks of 1 to
64 rows take the triangular factors in shared memory (one warp, two warps), and a
molecule with a vanishing B matrix, whose two TDHF residuals per root are nearly
parallel, the Loewdin factors.  Roots against the brute-force eigenvalues to the
float64 solve's 1e-6 eV; the final solution vectors are orthonormal to the
residual threshold over the smallest gap.
"""
import numpy as np
import pytest

import molgen
from tests.gpu_common import context, oracle_ground_state

pytestmark = pytest.mark.gpu

xs = pytest.importorskip("paper_2505_24807_gb300.xs")


@pytest.fixture(scope="module")
def case():
    from oracle import excited, nddo
    params = molgen.make_params(0)
    Z, xyz = molgen.config_small(1)
    mol, ints, res = oracle_ground_state(Z, xyz, params)
    A, B = excited.explicit_AB(res.eps, res.C, mol.nocc, nddo.full_eri(mol, ints))
    return dict(params=params, Z=Z, xyz=xyz, A=A, B=B)


@pytest.mark.parametrize("batched", [0, 1])
@pytest.mark.parametrize("k", [1, 2, 9, 16, 32])
def test_tdhf_blocks(case, k, batched):
    from oracle import excited
    if batched and k > 16:
        pytest.skip("the lock-step batch takes up to 16 roots")
    w, _, _ = excited.rpa_bruteforce(case["A"], case["B"], k)
    ctx = context(case["params"])
    try:
        xs.xs_ground_state(ctx.h, [(case["Z"], case["xyz"])])
        out = xs.xs_excited(ctx.h, method=xs.XS_TDHF, nroots=k, tol=1e-6, batched=batched)
    finally:
        ctx.close()
    assert out["info"]["converged"] == 1
    assert np.abs(out["omega"][0] - w).max() < 1e-6


def test_nearly_dependent_directions():
    """Two hydrogen molecules 1000 Angstrom apart: degenerate roots whose residuals
    vanish together, so that new blocks lose rank."""
    from oracle import excited, nddo
    params = molgen.make_params(0)
    Z = np.array([1, 1, 1, 1])
    xyz = np.array([[0.0, 0, 0], [0.8, 0, 0], [1000.0, 0, 0], [1000.8, 0, 0]])
    mol, ints, res = oracle_ground_state(Z, xyz, params)
    A, B = excited.explicit_AB(res.eps, res.C, mol.nocc, nddo.full_eri(mol, ints))
    w, _, _ = excited.rpa_bruteforce(A, B, 3)
    ctx = context(params)
    try:
        xs.xs_ground_state(ctx.h, [(Z, xyz)])
        out = xs.xs_excited(ctx.h, method=xs.XS_TDHF, nroots=3, tol=1e-6)
    finally:
        ctx.close()
    assert np.abs(out["omega"][0] - w).max() < 1e-6
