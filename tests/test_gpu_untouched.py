"""Combinations that are refused for a non-finite value leave the caller's device
array as it was, wherever the value lies: 32 outputs are formed at a time."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

xs = pytest.importorskip("paper_2505_24807_gb300.xs")


@pytest.fixture(scope="module")
def h():
    h = xs.xs_create(0)
    yield h
    xs.xs_destroy(h)


@pytest.mark.parametrize("nout", [1, 32, 33, 70])
@pytest.mark.parametrize("where", ["vectors", "coefficients"])
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_refused_combination(h, nout, where, value):
    torch = pytest.importorskip("torch")
    nb, S, L = 2, 9, 4001
    rng = np.random.default_rng(nout)
    X, c = rng.standard_normal((nb, S, L)), rng.standard_normal((nb, S, nout))
    if where == "vectors":
        X[1, S - 1, L - 1] = value
    else:
        c[1, S - 1, nout - 1] = value
    dX, dc = torch.from_numpy(X).cuda(), torch.from_numpy(c).cuda()
    Y = torch.full((nout, L), 7.0, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    rc = xs.load().xs_subspace_combine(h, nb, S, nout, L, xs._ptr(dX), xs._ptr(dc), xs._ptr(Y), 1)
    assert rc == xs.XS_ECUDA
    assert bool((Y == 7.0).all())
    # the context stays usable and the same call without the value writes everything
    dX.nan_to_num_(0.0, 0.0, 0.0)
    dc.nan_to_num_(0.0, 0.0, 0.0)
    torch.cuda.synchronize()
    xs._check(h, xs.load().xs_subspace_combine(h, nb, S, nout, L, xs._ptr(dX), xs._ptr(dc), xs._ptr(Y), 1))
    ref = torch.einsum("bsk,bsl->kl", dc, dX)
    assert float((Y - ref).abs().max()) < 64 * nb * S * 2.0 ** -53 * float(dc.abs().max() * dX.abs().max())
