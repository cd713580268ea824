"""Calls on two devices of one process, one after the other: a kernel's shared-memory
limit holds for the device that was current when it was set, so each device needs
its own, and scratch that outlives a call lies on the device that the call ran on."""
from tests import fake_cuda

SCRIPT = """
Z, xyz = molgen.make_chain(3, 40, 62)          # 222 AOs: residue products in float64
Zl, xyzl = molgen.make_chain(3, 110, 182)      # 622 AOs: float16 pairs in mixed precision
rng = np.random.default_rng(0)
def every_path(device):
    h = context(device)
    xs.xs_ground_state(h, [(Z, xyz), (Zl, xyzl)])
    for mol in (0, 1):
        n, o, _ = xs.xs_get_sizes(h, mol)
        X = rng.standard_normal((3, o * (n - o)))
        for precision in (xs.XS_FP64, xs.XS_MIXED):
            for kind in (xs.XS_KIND_A, xs.XS_KIND_APB, xs.XS_KIND_AMB, xs.XS_KIND_APB_TRIPLET):
                xs.xs_apply(h, mol, kind, X, precision=precision)
    for S in (10, 48, 100, 200, 224, 300):
        xs.xs_subspace_eig(h, np.eye(S), 10)
    for N in (5, 13, 21, 30, 40):
        xs.xs_subspace_gram(h, rng.standard_normal((12, 3000)), rng.standard_normal((N, 3000)))
        xs.xs_subspace_combine(h, rng.standard_normal((2, 12, 3000)), rng.standard_normal((2, 12, N)))
    for batched in (0, 1):
        for method in (xs.XS_CIS, xs.XS_TDHF):
            for precision in (xs.XS_FP64, xs.XS_MIXED):
                try:
                    xs.xs_excited(h, method=method, nroots=6, tol=1e-5, precision=precision, batched=batched)
                except xs.XSError as e:       # nothing converges here
                    assert e.status != xs.XS_ECUDA, e
    xs.xs_destroy(h)
every_path(0)
assert fake.fake_used(0) > 0 and fake.fake_used(1) == 0
every_path(1)
assert fake.fake_used(1) == fake.fake_used(0)
print("both devices")
"""


def test_second_device(tmp_path):
    assert "both devices" in fake_cuda.run(tmp_path, SCRIPT)
