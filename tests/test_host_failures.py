"""Every allocation of a call made to fail in turn, on the CPU against a stand-in for the
CUDA runtime: once (the call runs again by itself and succeeds where it gave anything
back) and from then on (it ends in XS_ENOMEM).  Whatever was left half-built must not
be taken for complete by the second run or by later calls."""
import pytest

from tests import fake_cuda

SCRIPT = """
small = molgen.make_chain(3, 12, 14)
large = molgen.make_chain(3, 100, 150)         # 550 AOs: float16 pairs in mixed precision
rng = np.random.default_rng(0)
def apply(mol, kind, precision):
    def call(h):
        n, o, _ = xs.xs_get_sizes(h, mol)
        xs.xs_apply(h, mol, kind, rng.standard_normal((2, o * (n - o))), precision=precision)
    return call
def solve(method, precision, batched, **more):
    def call(h):
        xs.xs_excited(h, method=method, nroots=3, tol=1e-6, max_iter=2, precision=precision, batched=batched, n_mol=2,
                      allow=(xs.XS_ENOCONV,), **more)   # no root of the batch converges here
    return call
def others(h):
    n, o, _ = xs.xs_get_sizes(h, 0)
    F, T = np.zeros((300, 11), np.float32), np.zeros((300, 2), np.float32)
    xs.xs_set_orbitals(h, 0, np.eye(n), np.arange(float(n)))
    xs.xs_get_orbitals(h, 0)
    xs.xs_subspace_eig(h, np.eye(300), 10)
    xs.xs_subspace_gram(h, rng.standard_normal((12, 3000)), rng.standard_normal((5, 3000)))
    xs.xs_subspace_combine(h, rng.standard_normal((2, 12, 3000)), rng.standard_normal((2, 12, 40)))
    xs.xs_mlp_init(h, 1)
    xs.xs_mlp_forward(h, F)
    xs.xs_mlp_train(h, F, T, 1, 100, 1e-3)
    xs.xs_excited(h, nroots=3, tol=1e-6, max_iter=2, guess=xs.XS_GUESS_LEARNED, n_mol=2)
    try:
        xs.xs_gradient(h, 0, 1)
    except xs.XSError as e:                    # no matrix is positive definite here
        if e.status != xs.XS_EUNSTABLE:
            raise
CALLS = {"apply": [apply(m, k, p) for m in (0, 1) for k in (xs.XS_KIND_A, xs.XS_KIND_APB) for p in (0, 1)],
         "solve": [solve(m, p, 0, subspace=s) for m in (0, 1) for p in (0, 1) for s in (1, 2)],
         "others": [others],
         "batch": [solve(m, p, 1) for m in (0, 1) for p in (0, 1)]}[WHAT]
mols = [small, large] if WHAT == "apply" else [small, small]
def roots_readable(h):
    for mol in range(2):
        n, o, _ = xs.xs_get_sizes(h, mol)
        try:
            xs.xs_get_amplitudes(h, mol, 0)
        except xs.XSError as e:
            assert e.status == xs.XS_ESTATE, e
def fail(call, after, times):
    # whether the call failed with `times` failing allocations after `after` good ones
    h = context()
    xs.xs_ground_state(h, mols)
    dipoles = fake.fake_launched(b"dipole_rc_kernel")
    fake.fake_fail(after, times)
    try:
        call(h)
        failed = False
    except xs.XSError as e:
        assert e.status == xs.XS_ENOMEM, (after, times, e)
        failed = True
    fake.fake_fail(-1, 0)
    roots_readable(h)
    call(h)
    roots_readable(h)
    if WHAT != "apply":                        # dipole integrals of both molecules, three components each
        built = fake.fake_launched(b"dipole_rc_kernel") - dipoles
        assert built >= 6, (after, times, built)
    xs.xs_destroy(h)
    return failed
for call in CALLS:
    count = 0
    while fail(call, count, 1 << 40):
        count += 1
    assert count > 3
    for after in range(count):
        fail(call, after, 1)
print("swept")
"""


@pytest.mark.parametrize("what", ["apply", "solve", "batch", "others"])
def test_every_allocation_fails_once(tmp_path, what):
    assert "swept" in fake_cuda.run(tmp_path, f"WHAT = {what!r}\n" + SCRIPT)
