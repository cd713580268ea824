"""Timed cases of libxs: the calls a program makes around a molecule's excited states.

A case is one call of the library's public interface (``paper_2505_24807_gb300.xs``)
on a molecule: the response products A X and (A +- B) X, the two-electron build G(R)
behind them and behind the Fock matrix, the float64 subspace products of the Davidson
step, the parameter gradient of a root, and three whole solves.  The molecules are the
seeded chains of ``molgen`` (the benchmark's small, medium and large ones and odd sizes
between them), moved by a thermal jitter that depends on the seed, as the frames of a
dynamics run differ.
"""
import functools
import itertools
import math

import numpy as np
import torch

import molgen
from paper_2505_24807_gb300 import xs

KAPPA = 14.399645          # e^2 / (4 pi eps0), eV Angstrom
HARTREE, BOHR = 27.211386245988, 0.529177210903
CORE = {1: 1.0, 6: 4.0, 7: 5.0, 8: 6.0}
PAIRS = [(0, 0), (0, 1), (0, 2), (0, 3), (1, 1), (1, 2), (1, 3), (2, 2), (2, 3), (3, 3)]
PROD = [[next(k for k, p in enumerate(PAIRS) if p == (min(m, n), max(m, n))) for n in range(4)] for m in range(4)]
KINDS = {"A": xs.XS_KIND_A, "A+B": xs.XS_KIND_APB, "A-B": xs.XS_KIND_AMB, "A triplet": xs.XS_KIND_A_TRIPLET,
         "A+B triplet": xs.XS_KIND_APB_TRIPLET}
JITTER = 0.01              # Angstrom: the spread of a frame's coordinates around the chain
MAX_DENSE = 4000           # largest nocc * nvir that exact() diagonalises


def listed():
    return [
        # a small molecule's CIS product: a few launches on 62 AOs, all latency
        dict(name="cis_product_small", op="product", kind="A", precision="f64", heavy=12, h=14, nvec=5),
        # a ragged molecule's second TDHF product, a part of a block of vectors left unconverged
        dict(name="tdhf_product_ragged", op="product", kind="A-B", precision="f64", heavy=97, h=191, nvec=7),
        # the float64 reference product of the largest molecule, one block of four vectors
        dict(name="tdhf_product_large", op="product", kind="A+B", precision="f64", heavy=400, h=600, nvec=4),
        # ten roots' block of a medium molecule in the mixed precision that solves use
        dict(name="cis_product_mixed", op="product", kind="A", precision="mixed", heavy=100, h=200, nvec=10),
        # the block that dominates a large TDHF solve: two vectors for each of ten roots
        dict(name="tdhf_product_mixed_large", op="product", kind="A+B", precision="mixed", heavy=400, h=600, nvec=20),
        # two-electron build of a few AO densities (Fock matrices, difference densities)
        dict(name="two_electron_build", op="gbuild", precision="f64", heavy=233, h=301, nvec=4),
        # projections of a Davidson block onto the subspace
        dict(name="subspace_projection", op="gram", s=120, new=20, length=373100),
        # Ritz vectors and residuals out of the subspace
        dict(name="subspace_combination", op="combine", blocks=2, s=120, new=20, length=179400),
        # the backward direction: d omega / d parameter of a root, orbital response included
        dict(name="parameter_gradient", op="gradient", method="cis", heavy=60, h=91, roots=5, root=0),
        # whole solve of a small molecule in float64
        dict(name="cis_solve_small", op="solve", method="cis", precision="f64", heavy=12, h=14, roots=5),
        # whole TDHF solve of a medium molecule in mixed precision
        dict(name="tdhf_solve_medium", op="solve", method="tdhf", precision="mixed", heavy=100, h=200, roots=10),
        # sixteen molecules of uneven size in the lock-step batch
        dict(name="cis_solve_batch", op="batch", method="cis", precision="mixed", molecules=16, most_atoms=140, roots=6),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def hydrogens(heavy):
        return int(round(heavy * rng.uniform(1.4, 1.8)))

    op = rng.choice(["product"] * 6 + ["gbuild", "gram", "combine", "gradient", "solve", "batch"])
    if op == "product":
        precision = rng.choice(["f64", "mixed"])
        heavy = log(10, 300)
        # the block shrinks with the molecule so that no draw costs more than the large listed products
        most = max(1, min(20, int((4 if precision == "f64" else 20) * (400.0 / heavy) ** 3 / 3)))
        return dict(op=op, kind=rng.choice(sorted(KINDS)), precision=precision, heavy=heavy, h=hydrogens(heavy),
                    nvec=rng.randint(1, most))
    if op == "gbuild":
        heavy = log(12, 300)
        return dict(op=op, precision="f64", heavy=heavy, h=hydrogens(heavy), nvec=rng.randint(1, 6))
    if op == "gram":
        return dict(op=op, s=log(8, 150), new=rng.randint(1, 24), length=log(1000, 373100))
    if op == "combine":
        return dict(op=op, blocks=rng.randint(1, 3), s=log(8, 110), new=rng.randint(1, 24), length=log(1000, 179400))
    if op == "gradient":
        heavy = log(8, 60)
        roots = rng.randint(2, 5)
        return dict(op=op, method=rng.choice(["cis", "tdhf"]), heavy=heavy, h=hydrogens(heavy), roots=roots,
                    root=rng.randrange(roots))
    if op == "solve":
        precision = rng.choice(["f64", "mixed"])
        heavy = log(8, 16) if precision == "f64" else log(12, 100)
        return dict(op=op, method=rng.choice(["cis", "tdhf"]), precision=precision, heavy=heavy, h=hydrogens(heavy),
                    roots=rng.randint(2, 8))
    return dict(op=op, method="cis", precision="mixed", molecules=rng.randint(4, 16), most_atoms=rng.randint(40, 140),
                roots=rng.randint(3, 6))


# ---- inputs -----------------------------------------------------------------------------------

PARAMS = molgen.make_params(0)


@functools.lru_cache(maxsize=None)
def _stream():
    return torch.cuda.Stream()


@functools.lru_cache(maxsize=64)
def _chain(heavy, h):
    """The chain of these counts (the next hydrogen count that closes the shells, if this one does not)."""
    for more in range(4):
        for seed in range(3):
            try:
                Z, xyz = molgen.make_chain(heavy + seed, heavy, h + more)
                if sum(int(CORE[int(z)]) for z in Z) % 2 == 0:
                    return np.asarray(Z), np.asarray(xyz)
            except (ValueError, RuntimeError):
                continue
    raise ValueError("no chain of %d heavy atoms and %d hydrogens" % (heavy, h))


def _frame(heavy, h, seed):
    Z, xyz = _chain(heavy, h)
    return Z, xyz + JITTER * np.random.default_rng(seed).uniform(-1.0, 1.0, xyz.shape)


def _layout(Z):
    """Padded position (4 per atom) of every AO, and the number of occupied orbitals."""
    pos = [4 * a + k for a, z in enumerate(Z) for k in range(1 if z == 1 else 4)]
    return torch.tensor(pos, device="cuda"), int(sum(CORE[int(z)] for z in Z)) // 2


def _atom(Z, field):
    return torch.tensor([PARAMS[int(z)][field] for z in Z], dtype=torch.float64, device="cuda")


def _resonance(Z, xyz):
    """Off-diagonal part of the core Hamiltonian, (beta_mu + beta_lam) / 2 times the overlap, 4 rows per atom."""
    x = torch.as_tensor(xyz, device="cuda")
    N = len(Z)
    d = x[None, :, :] - x[:, None, :]
    eye = torch.eye(N, dtype=torch.float64, device="cuda")
    r = torch.sqrt((d * d).sum(-1) + eye)
    e = d / r[:, :, None]
    zs, zp = _atom(Z, "zeta_s"), _atom(Z, "zeta_p")

    def radial(a, za, zb, scale=1.0):
        return a * torch.exp(-scale * 0.5 * (za[:, None] + zb[None, :]) * r) * (1.0 - eye)

    S = torch.zeros(N, 4, N, 4, dtype=torch.float64, device="cuda")
    S[:, 0, :, 0] = radial(2.0, zs, zs)
    S[:, 0, :, 1:] = -e * radial(2.4, zs, zp)[:, :, None]
    S[:, 1:, :, 0] = (e * radial(2.4, zp, zs)[:, :, None]).transpose(1, 2)
    sig, pi = radial(1.9, zp, zp), radial(1.6, zp, zp, 1.3)
    ee = e[:, :, :, None] * e[:, :, None, :]
    pp = -ee * sig[:, :, None, None] + (torch.eye(3, dtype=torch.float64, device="cuda") - ee) * pi[:, :, None, None]
    S[:, 1:, :, 1:] = pp.permute(0, 2, 1, 3)
    beta = torch.stack([_atom(Z, "beta_s")] + [_atom(Z, "beta_p")] * 3, 1).reshape(-1)
    return 0.5 * (beta[:, None] + beta[None, :]) * S.reshape(4 * N, 4 * N)


def _product_inputs(case, seed):
    """Geometry, the caller's own orbitals (of the resonance Hamiltonian with atomic levels on its diagonal) and a
    block of normalised trial vectors weighted by their gaps like preconditioned residuals."""
    Z, xyz = _frame(case["heavy"], case["h"], seed)
    pos, o = _layout(Z)
    F = _resonance(Z, xyz)
    level = torch.tensor([[-12.0] * 4 if z == 1 else [-18.0 - z] + [-6.0 - z] * 3 for z in Z], dtype=torch.float64, device="cuda")
    F = (F + torch.diag(level.reshape(-1)))[pos][:, pos]
    eps, C = torch.linalg.eigh(0.5 * (F + F.T))
    g = torch.Generator(device="cuda").manual_seed(seed)
    gap = eps[None, o:] - eps[:o, None]
    X = torch.randn(case["nvec"], *gap.shape, generator=g, dtype=torch.float64, device="cuda") / (1.0 + gap - gap.min())
    X = X.reshape(case["nvec"], -1)
    return Z, xyz, pos, o, C.contiguous(), eps, X / X.norm(dim=1, keepdim=True)


def _densities(case, seed):
    Z, xyz = _frame(case["heavy"], case["h"], seed)
    pos, _ = _layout(Z)
    n = len(pos)
    g = torch.Generator(device="cuda").manual_seed(seed)
    U = torch.randn(case["nvec"], n, 24, generator=g, dtype=torch.float64, device="cuda") / math.sqrt(n)
    return Z, xyz, pos, U @ U.transpose(1, 2) + torch.diag(torch.full((n,), 0.5, dtype=torch.float64, device="cuda"))


def _subspace(case, seed):
    """Rows of a Davidson subspace: unit rows over the amplitudes, with coefficients of that size."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    L = case["length"]
    if case["op"] == "gram":
        A, B = (torch.randn(k, L, generator=g, dtype=torch.float64, device="cuda") / math.sqrt(L)
                for k in (case["s"], case["new"]))
        return A, B
    X = torch.randn(case["blocks"], case["s"], L, generator=g, dtype=torch.float64, device="cuda") / math.sqrt(L)
    c = torch.randn(case["blocks"], case["s"], case["new"], generator=g, dtype=torch.float64, device="cuda")
    return X, c / math.sqrt(case["s"])


class State:
    """A library context on the program's stream, closed with the state, and the call's arrays."""

    def __init__(self, case):
        self.case = case
        self.ctx = xs.xs_create(0, stream=_stream().cuda_stream)
        xs.xs_set_params(self.ctx, molgen.params_table(PARAMS))

    def __del__(self):
        if getattr(self, "ctx", None) is not None:
            xs.xs_destroy(self.ctx)
            self.ctx = None


METHOD = {"cis": xs.XS_CIS, "tdhf": xs.XS_TDHF}
PRECISION = {"f64": xs.XS_FP64, "mixed": xs.XS_MIXED}


def prepare(case, seed):
    torch.zeros(1, device="cuda")
    with torch.cuda.stream(_stream()):
        st = State(case)
        op = case["op"]
        if op == "product":
            Z, xyz, _, _, C, eps, st.X = _product_inputs(case, seed)
            # integrals and layout; the orbitals are the caller's own, so the first SCF step is enough
            xs.xs_ground_state(st.ctx, [(Z, xyz)], scf_tol=1e6)
            xs._check(st.ctx, xs.load().xs_set_orbitals(st.ctx, 0, xs._ptr(C), xs._ptr(eps)))
        elif op == "gbuild":
            Z, xyz, _, st.X = _densities(case, seed)
            xs.xs_ground_state(st.ctx, [(Z, xyz)], scf_tol=1e6)
        elif op in ("gram", "combine"):
            st.X, st.Y = _subspace(case, seed)
            rows, cols = (case["s"], case["new"]) if op == "gram" else (case["new"], case["length"])
            st.out = torch.empty(rows, cols, dtype=torch.float64, device="cuda")
        else:
            if op == "batch":
                sizes = np.random.default_rng(7).integers(20, case["most_atoms"] + 1, case["molecules"])
                mols = [_frame(max(1, round(0.4 * int(a))), int(a) - max(1, round(0.4 * int(a))), seed + k)
                        for k, a in enumerate(sizes)]
            else:
                mols = [_frame(case["heavy"], case["h"], seed)]
            xs.xs_ground_state(st.ctx, mols)
            st.count = len(mols)
            if op == "gradient":
                xs.xs_excited(st.ctx, method=METHOD[case["method"]], nroots=case["roots"], tol=1e-8)
        _stream().synchronize()
    return st


def run(st):
    case = st.case
    op = case["op"]
    with torch.cuda.stream(_stream()):
        if op == "product":
            Y = xs.xs_apply(st.ctx, 0, KINDS[case["kind"]], st.X, precision=PRECISION[case["precision"]])
            # a mixed product carries float32 accuracy, and its caller keeps it so
            return Y if case["precision"] == "f64" else Y.to(torch.float32)
        if op == "gbuild":
            return xs.xs_apply(st.ctx, 0, xs.XS_KIND_G, st.X)
        if op == "gram":
            xs._check(st.ctx, xs.load().xs_subspace_gram(st.ctx, case["s"], case["new"], case["length"], xs._ptr(st.X),
                                                         xs._ptr(st.Y), xs._ptr(st.out), 1))
            return st.out
        if op == "combine":
            xs._check(st.ctx, xs.load().xs_subspace_combine(st.ctx, case["blocks"], case["s"], case["new"],
                                                            case["length"], xs._ptr(st.X), xs._ptr(st.Y),
                                                            xs._ptr(st.out), 1))
            return st.out
        if op == "gradient":
            return xs.xs_gradient(st.ctx, 0, case["root"])[0]
        mixed = case["precision"] == "mixed"
        r = xs.xs_excited(st.ctx, method=METHOD[case["method"]], nroots=case["roots"], tol=1e-5 if mixed else 1e-6,
                          precision=PRECISION[case["precision"]], batched=1 if op == "batch" else 0, n_mol=st.count)
    if mixed:
        # a mixed solve stops at a 1e-4 eV residual: its energies (quadratic in it) are float32-grade numbers, its
        # strengths (linear in it) are fixed only to the third digit
        return r["omega"].astype(np.float32)
    return r["omega"], r["osc"]


# ---- work -------------------------------------------------------------------------------------

def _sizes(heavy, h):
    Z, _ = _chain(heavy, h)
    n = int(sum(1 if z == 1 else 4 for z in Z))
    o = int(sum(CORE[int(z)] for z in Z)) // 2
    return n, o, n - o, int(sum(1 if z == 1 else 10 for z in Z))


def _product_work(n, o, v, npr, nvec, real=8):
    """P build, two-electron build and back-transform of nvec vectors; every integral read once."""
    m = min(o, v)
    flops = nvec * (2 * (2.0 * n * o * v + 2.0 * n * n * m) + 32.0 * n * n + 2.0 * npr * npr)
    return dict(bytes=16.0 * nvec * o * v + real * (n * n + npr * npr / 2.0), flops=flops)


def work(case):
    op = case["op"]
    if op == "gram":
        s, k, L = case["s"], case["new"], case["length"]
        return dict(bytes=8.0 * ((s + k) * L + s * k), flops=2.0 * s * k * L)
    if op == "combine":
        s, k, L = case["blocks"] * case["s"], case["new"], case["length"]
        return dict(bytes=8.0 * ((s + k) * L + s * k), flops=2.0 * s * k * L)
    if op == "gbuild":
        n, _, _, npr = _sizes(case["heavy"], case["h"])
        return dict(bytes=case["nvec"] * 16.0 * n * n + 4.0 * npr * npr,
                    flops=case["nvec"] * (32.0 * n * n + 2.0 * npr * npr))
    if op == "batch":
        sizes = np.random.default_rng(7).integers(20, case["most_atoms"] + 1, case["molecules"])
        total = dict(bytes=0.0, flops=0.0)
        for a in sizes:
            heavy = max(1, round(0.4 * int(a)))
            one = _product_work(*_sizes(heavy, int(a) - heavy), 3 * case["roots"], 4)
            total = {k: total[k] + one[k] for k in total}
        return total
    size = _sizes(case["heavy"], case["h"])
    if op == "product":
        return _product_work(*size, case["nvec"], 8 if case["precision"] == "f64" else 4)
    if op == "gradient":
        return _product_work(*size, 10)      # the adjoint solve's products
    return _product_work(*size, 3 * case["roots"], 8 if case["precision"] == "f64" else 4)   # guess block and one more


# ---- the same numbers in plain float64 ------------------------------------------------------------

def _matchings(m):
    pairs = list(itertools.combinations(range(m), 2))
    for r in range(m // 2 + 1):
        for combo in itertools.combinations(pairs, r):
            used = [p for pr in combo for p in pr]
            if len(set(used)) == len(used):
                yield combo, [p for p in range(m) if p not in used]


class Model:
    """Two-centre product integrals W (atoms x atoms x 10 x 10, zero on the diagonal) and one-centre tensors of a
    molecule; a hydrogen's unused products meet zero rows of the padded densities."""

    def __init__(self, Z, xyz):
        self.Z = Z
        self.pos, self.o = _layout(Z)
        self.n, N = len(self.pos), len(Z)
        x = torch.as_tensor(xyz, device="cuda")
        d = (x[None, :, :] - x[:, None, :]).permute(2, 0, 1)
        eye = torch.eye(N, dtype=torch.float64, device="cuda")
        r = torch.sqrt((d * d).sum(0) + eye)
        sigma = KAPPA / (math.sqrt(math.pi) * _atom(Z, "gss"))
        a = 1.0 / torch.sqrt(2.0 * (sigma[:, None] ** 2 + sigma[None, :] ** 2))
        b = [torch.erf(a * r) / r]
        for k in range(1, 5):
            b.append(((2 * k - 1) * b[-1] - (2 * a * a) ** k / (a * math.sqrt(math.pi)) * torch.exp(-(a * r) ** 2)) / r ** 2)
        g = [(-1) ** k * KAPPA * b[k] * (1.0 - eye) for k in range(5)]

        @functools.lru_cache(maxsize=None)
        def deriv(idx):
            t = torch.zeros_like(r)
            for pairs, singles in _matchings(len(idx)):
                if all(idx[i] == idx[j] for i, j in pairs):
                    term = g[len(idx) - len(pairs)].clone()
                    for q in singles:
                        term = term * d[idx[q]]
                    t += term
            return t

        D1, D2 = _atom(Z, "D1"), _atom(Z, "D2")
        one = torch.ones(N, dtype=torch.float64, device="cuda")
        terms = []
        for m, k in PAIRS:
            if k == 0:
                terms.append([((), one)])
            elif m == 0:
                terms.append([((k - 1,), -D1)])
            else:
                terms.append(([((), one)] if m == k else []) + [((m - 1, k - 1), D2 * D2)])
        self.W = torch.zeros(N, N, 10, 10, dtype=torch.float64, device="cuda")
        for p in range(10):
            for q in range(10):
                for ia, ca in terms[p]:
                    for ib, cb in terms[q]:
                        self.W[:, :, p, q] += ca[:, None] * cb[None, :] * (-1) ** len(ib) * deriv(tuple(sorted(ia + ib)))
        P = torch.tensor(PROD, device="cuda")
        # exchange of block (A, B): K[m, l] = sum_{n, s} (m n | l s) R[n, s]
        i = torch.arange(4, device="cuda")
        m_, l_, n_, s_ = (i.view([-1 if k == j else 1 for k in range(4)]) for j in range(4))
        self.X = self.W[:, :, P[m_, n_], P[l_, s_]].reshape(N, N, 16, 16)
        self.P = P.reshape(-1)
        t = torch.zeros(N, 4, 4, 4, 4, dtype=torch.float64)
        for k, z in enumerate(Z):
            p = PARAMS[int(z)]
            t[k, 0, 0, 0, 0] = p["gss"]
            if z == 1:
                continue
            hpp = 0.5 * (p["gpp"] - p["gp2"])
            for u in range(1, 4):
                t[k, 0, 0, u, u] = t[k, u, u, 0, 0] = p["gsp"]
                t[k, u, u, u, u] = p["gpp"]
                t[k, 0, u, 0, u] = t[k, 0, u, u, 0] = t[k, u, 0, 0, u] = t[k, u, 0, u, 0] = p["hsp"]
                for w in range(1, 4):
                    if u != w:
                        t[k, u, u, w, w] = p["gp2"]
                        t[k, u, w, u, w] = t[k, u, w, w, u] = hpp
        self.T = t.cuda()

    def jk(self, R):
        """J(R) and K(R) of one n x n matrix."""
        N = len(self.Z)
        full = torch.zeros(4 * N, 4 * N, dtype=torch.float64, device="cuda")
        full[self.pos[:, None], self.pos[None, :]] = R
        B = full.reshape(N, 4, N, 4).permute(0, 2, 1, 3)                 # atom, atom, ao, ao
        diag = B[torch.arange(N), torch.arange(N)]
        r = torch.zeros(N, 10, dtype=torch.float64, device="cuda").index_add_(1, self.P, diag.reshape(N, 16))
        j2 = torch.einsum("abpq,bq->ap", self.W, r)[:, self.P].reshape(N, 4, 4)
        J = torch.zeros(N, N, 4, 4, dtype=torch.float64, device="cuda")
        K = torch.matmul(self.X, B.reshape(N, N, 16, 1)).reshape(N, N, 4, 4)
        k = torch.arange(N)
        J[k, k] = j2 + torch.einsum("amnls,als->amn", self.T, diag)
        K[k, k] = torch.einsum("amlns,als->amn", self.T, diag)
        return tuple(M.permute(0, 2, 1, 3).reshape(4 * N, 4 * N)[self.pos][:, self.pos] for M in (J, K))

    def product(self, kind, C, eps, X):
        o = self.o
        out = []
        gap = eps[None, o:] - eps[:o, None]
        for x in X:
            x = x.reshape(gap.shape)
            J, K = self.jk(C[:, :o] @ x @ C[:, o:].T)
            # K of the transposed density is the transpose of K
            G = {"A": 2 * J - K, "A+B": 4 * J - K - K.T, "A-B": K.T - K, "A triplet": -K, "A+B triplet": -K - K.T}[kind]
            out.append((gap * x + C[:, :o].T @ G @ C[:, o:]).reshape(-1))
        return torch.stack(out)

    def core(self, xyz):
        N = len(self.Z)
        H = _resonance(self.Z, xyz).reshape(N, 4, N, 4)
        z = torch.tensor([CORE[int(q)] for q in self.Z], dtype=torch.float64, device="cuda")
        att = torch.einsum("abp,b->ap", self.W[:, :, :, 0], z)[:, self.P].reshape(N, 4, 4)
        k = torch.arange(N)
        level = torch.stack([_atom(self.Z, "Uss")] + [_atom(self.Z, "Upp")] * 3, 1)
        H[k, :, k, :] += torch.diag_embed(level) - att
        return H.reshape(4 * N, 4 * N)[self.pos][:, self.pos]

    def ground_state(self, xyz):
        H, o, n = self.core(xyz), self.o, self.n
        occ = [CORE[int(z)] / (1 if z == 1 else 4) for z in self.Z for _ in range(1 if z == 1 else 4)]
        D = torch.diag(torch.tensor(occ, dtype=torch.float64, device="cuda"))
        Fs, Es = [], []
        for _ in range(200):
            J, K = self.jk(D)
            F = H + J - 0.5 * K
            E = F @ D - D @ F
            Fs, Es = (Fs + [F])[-10:], (Es + [E])[-10:]
            m = len(Fs)
            B = -torch.ones(m + 1, m + 1, dtype=torch.float64)
            B[m, m] = 0.0
            for i in range(m):
                for j in range(m):
                    B[i, j] = float((Es[i] * Es[j]).sum())
            rhs = torch.zeros(m + 1, dtype=torch.float64)
            rhs[m] = -1.0
            if m > 1:
                scale = float(B[:m, :m].abs().max())
                B[:m, :m] /= scale
                c = torch.linalg.solve(B, rhs)[:m]
                F = sum(float(ci) * Fi for ci, Fi in zip(c, Fs))
            eps, C = torch.linalg.eigh(F)
            new = 2.0 * C[:, :o] @ C[:, :o].T
            done = float((new - D).abs().max()) < 1e-11 and float(E.abs().max()) < 1e-10
            D = new
            if done:
                break
        J, K = self.jk(D)
        return torch.linalg.eigh(H + J - 0.5 * K)

    def roots(self, xyz, method, k):
        """Lowest k energies and oscillator strengths from the explicit matrices."""
        eps, C = self.ground_state(xyz)
        o, ov = self.o, self.o * (self.n - self.o)
        one = torch.eye(ov, dtype=torch.float64, device="cuda")
        if method == "cis":
            w, U = torch.linalg.eigh(self.product("A", C, eps, one))
            w, U = w[:k], U[:, :k]
        else:
            plus, minus = self.product("A+B", C, eps, one), self.product("A-B", C, eps, one)
            Lo = torch.linalg.cholesky(0.5 * (minus + minus.T))
            w, V = torch.linalg.eigh(Lo.T @ (0.5 * (plus + plus.T)) @ Lo)
            w = torch.sqrt(w[:k])
            U = Lo @ V[:, :k] / torch.sqrt(w)
        dip = torch.zeros(3, 4 * len(self.Z), 4 * len(self.Z), dtype=torch.float64)
        for a, z in enumerate(self.Z):
            for x in range(3):
                for q in range(4):
                    dip[x, 4 * a + q, 4 * a + q] = float(xyz[a][x])
                dip[x, 4 * a, 4 * a + 1 + x] = dip[x, 4 * a + 1 + x, 4 * a] = PARAMS[int(z)]["D1"]
        dip = dip.cuda()[:, self.pos][:, :, self.pos]
        mo = (C[:, :o].T @ dip @ C[:, o:]).reshape(3, ov)
        t = math.sqrt(2.0) * mo @ U / BOHR
        return w, (2.0 / 3.0) * (w / HARTREE) * (t * t).sum(0)


def exact(case, seed):
    op = case["op"]
    if op == "product":
        Z, xyz, _, _, C, eps, X = _product_inputs(case, seed)
        return Model(Z, xyz).product(case["kind"], C, eps, X)
    if op == "gbuild":
        Z, xyz, _, R = _densities(case, seed)
        m = Model(Z, xyz)
        return torch.stack([2 * J - K for J, K in map(m.jk, R)])
    if op == "gram":
        A, B = _subspace(case, seed)
        return A @ B.T
    if op == "combine":
        X, c = _subspace(case, seed)
        return torch.einsum("bsk,bsl->kl", c, X)
    if op == "solve":
        n, o, v, _ = _sizes(case["heavy"], case["h"])
        if o * v > MAX_DENSE:
            return None
        Z, xyz = _frame(case["heavy"], case["h"], seed)
        w, f = Model(Z, xyz).roots(xyz, case["method"], case["roots"])
        return w[None, :] if case["precision"] == "mixed" else (w[None, :], f[None, :])
    return None      # the gradient differentiates the whole model; the batch's larger molecules are not diagonalised
