"""Performance cases of the library: what a user's program has it do.

A replica-parallel simulation step (path-integral MD beads, string images) is
one forces call for all replicas; the call's blocks are the Fock build of a
given density and the batched diagonalisation, each callable by itself; the
learned starting density has its training step. The cases run these public
entry points over the range of the repository's own workloads: water clusters
of 1 to 16 molecules in the minimal and the split-valence basis, Diels-Alder
images, FP64 and the mixed-precision mode.

listed() / draw(rng) give cases, prepare(case, seed) what a program has in
hand before the call, run(state) one pass, work(case) the bytes and operations
that the path cannot do without, exact(case, seed) the outputs in 64 bits from
plain torch, without the library.
"""
import math

import numpy as np
import torch

from paper_1601_02713_gb300 import inputs, native

_ctx = None
_bases = {}


def _context():
    """The one context a program keeps."""
    global _ctx
    if _ctx is None:
        _ctx = native.Context(0)
    return _ctx


def _basis(kind):
    if kind not in _bases:
        _bases[kind] = native.Basis(inputs.basis_set(kind))
    return _bases[kind]


def listed():
    return [
        # the smallest forces call: 4 beads of the water dimer in the minimal
        # basis (14 functions), FP64, from the core Hamiltonian
        dict(name="forces_dimer_min", kind="forces", nwater=2, basis="min_sp", beads=4, fp32_tau=0.0, guess=0),
        # two consecutive MD steps of 4 beads of the dimer in the s/p/d basis:
        # SAD, then the previous step's MOs
        dict(name="md_dimer_spd", kind="md", nwater=2, basis="split_spd", beads=4, fp32_tau=0.0, steps=2),
        # string images of uneven size (1 to 4 waters) in one ragged call
        dict(name="images_ragged_spd", kind="images", nmax=4, basis="split_spd", images=5, fp32_tau=0.0, guess=4),
        # one bead of (H2O)8, the benchmark's cluster (192 functions), FP64
        dict(name="forces_water8_fp64", kind="forces", nwater=8, basis="split_spd", beads=1, fp32_tau=0.0, guess=4),
        # a bead of a smaller cluster in the mixed-precision mode
        dict(name="forces_water6_mixed", kind="forces", nwater=6, basis="split_spd", beads=1, fp32_tau=1e-6, guess=4),
        # Fock builds of a given density: the smallest molecule (24 functions)
        dict(name="fock_water1", kind="fock", system="water", size=1, basis="split_spd", beads=1, fp32_tau=0.0),
        # 4 beads of (H2O)8 in one batch, FP64 (the step's dominating kernels)
        dict(name="fock_water8_batch", kind="fock", system="water", size=8, basis="split_spd", beads=4, fp32_tau=0.0),
        # a Diels-Alder image with 3 waters (C, O and H, 272 functions)
        dict(name="fock_diels_alder", kind="fock", system="da", size=3, basis="split_spd", beads=1, fp32_tau=0.0),
        # the largest: (H2O)16, 384 functions
        dict(name="fock_water16", kind="fock", system="water", size=16, basis="split_spd", beads=1, fp32_tau=0.0),
        # diagonalisation of an SCF iteration: 32 beads of 192 functions
        dict(name="eigh_192", kind="eigh", n=192, nmat=32),
        # a training step of the learned density (oxygen pairs of 32 beads of (H2O)8)
        dict(name="train_guess_oo", kind="train", type=3, rows=896),
    ]


def draw(rng):
    kind = rng.choice(["forces", "md", "images", "fock", "fock", "eigh", "train"])

    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    tau = rng.choice([0.0, 0.0, 1e-6])
    if kind == "forces":
        if rng.random() < 0.4:
            return dict(kind=kind, nwater=logint(1, 8), basis="min_sp", beads=logint(1, 32), fp32_tau=tau, guess=4)
        n = logint(1, 6)
        return dict(kind=kind, nwater=n, basis="split_spd", beads=logint(1, max(1, 24 // n ** 2)), fp32_tau=tau,
                    guess=rng.choice([0, 4]))
    if kind == "md":
        n = logint(1, 3)
        return dict(kind=kind, nwater=n, basis=rng.choice(["min_sp", "split_spd"]), beads=logint(1, 12 // n ** 2 + 1),
                    fp32_tau=tau, steps=rng.randint(2, 3))
    if kind == "images":
        return dict(kind=kind, nmax=rng.randint(2, 4), basis="split_spd", images=rng.randint(2, 7), fp32_tau=tau,
                    guess=4)
    if kind == "fock":
        if rng.random() < 0.25:
            return dict(kind=kind, system="da", size=rng.randint(0, 4), basis="split_spd", beads=1, fp32_tau=tau)
        n = logint(1, 16)
        return dict(kind=kind, system="water", size=n, basis="split_spd", beads=logint(1, max(1, 192 // n ** 2)),
                    fp32_tau=tau)
    if kind == "eigh":
        n = logint(7, 384)
        return dict(kind=kind, n=n, nmat=logint(1, max(1, min(64, 3000000 // n ** 3 * 8 + 1))))
    return dict(kind=kind, type=rng.randint(0, 8), rows=logint(32, 4096))


# ---------------------------------------------------------------- inputs
def _molecule(system, size, seed):
    """(Z, coords in Angstrom) of a seeded geometry."""
    if system == "da":
        reps = inputs.diels_alder_images(24, 4)
        k = size + 5 * (seed % 4)   # an image with `size` waters
        return reps.Z[k], reps.coords[k] / inputs.ANGSTROM_TO_BOHR
    if size == 2:
        return inputs.water_dimer_geometry(seed % 1000 + 1)
    return inputs.water_cluster_geometry(size, seed % 1000 + 2)


def _beads(system, size, nrep, seed):
    Z, xyz = _molecule(system, size, seed)
    return inputs.beads(Z, xyz, nrep, 2000 + 64 * (seed % 100003))


def _atom_of_function(Z, kind):
    bas = inputs.basis_set(kind)
    return np.concatenate([np.full(sum(2 * s.l + 1 for s in bas[int(z)]), a) for a, z in enumerate(Z)])


def _density(Z, X, kind, rng):
    """A density of SCF-like form: doubly occupied orbitals, each centred on an
    atom and decaying with the distance from it, tr D = number of electrons."""
    at = _atom_of_function(Z, kind)
    nocc = int(Z.sum()) // 2
    centre = rng.choice(len(Z), nocc, p=Z / Z.sum())
    d = np.linalg.norm(X[at][:, None, :] - X[centre][None, :, :], axis=-1)
    C = rng.normal(size=(len(at), nocc)) * np.exp(-d / 1.5)
    C /= np.linalg.norm(C, axis=0)
    return 2.0 * C @ C.T


def _symmetric(nmat, n, seed):
    """Fock-like symmetric matrices: nearly diagonal spectrum of the size of
    orbital energies with smaller couplings."""
    rng = np.random.default_rng(seed)
    A = rng.normal(size=(nmat, n, n)) * 0.1
    A = 0.5 * (A + A.transpose(0, 2, 1))
    A[:, range(n), range(n)] += np.sort(rng.uniform(-20.0, 30.0, size=(nmat, n)), axis=1)
    return A


def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng(seed)
    if kind in ("forces", "md"):
        reps = _beads("water", case["nwater"], case["beads"], seed)
        steps = inputs.markov_steps(reps, case.get("steps", 1), seed % 9973)
        Z, _ = reps.stacked()
        X = [torch.tensor(s.stacked()[1], device="cuda") for s in steps]
        opts = native.scf_opts(guess=case.get("guess", 5), fp32_tau=case["fp32_tau"])
        return dict(case=case, ctx=_context(), basis=_basis(case["basis"]), Z=Z, X=X, opts=opts)
    if kind == "images":
        Zs, Xs = [], []
        for i in range(case["images"]):
            r = _beads("water", 1 + i % case["nmax"], 1, seed + 7 * i)
            Zs.append(r.Z[0])
            Xs.append(r.coords[0])
        nat = np.array([len(z) for z in Zs], np.int32)
        opts = native.scf_opts(guess=case["guess"], fp32_tau=case["fp32_tau"])
        return dict(case=case, ctx=_context(), basis=_basis(case["basis"]), nat=nat, Z=np.concatenate(Zs),
                    X=torch.tensor(np.concatenate(Xs), device="cuda"), opts=opts)
    if kind == "fock":
        Z, X = _beads(case["system"], case["size"], case["beads"], seed).stacked()
        D = np.stack([_density(Z, x, case["basis"], rng) for x in X])
        return dict(case=case, ctx=_context(), basis=_basis(case["basis"]), Z=Z, X=X,
                    D=torch.tensor(D, device="cuda"))
    if kind == "eigh":
        A = torch.tensor(_symmetric(case["nmat"], case["n"], seed), device="cuda")
        return dict(case=case, ctx=_context(), A=A)
    # training rows of the pair type: random features of the size the
    # featuriser gives, density-like targets
    model = native.GuessModel(_basis("split_spd"), seed=seed % 1000)
    na, nb = _head(case["type"])
    Xf = np.zeros((case["rows"], 96), np.float32)
    Xf[:, :80] = rng.uniform(0.0, 1.0, size=(case["rows"], 80))
    Yf = (0.2 * rng.normal(size=(case["rows"], na * nb))).astype(np.float32)
    return dict(case=case, model=model, X=Xf, Y=Yf)


def _head(type_):
    """Functions of the two atoms of a pair type (0..2 one atom H, C, O; 3..8 OO, OC, OH, CC, CH, HH)."""
    return [(5, 5), (14, 14), (14, 14), (14, 14), (14, 14), (14, 5), (14, 14), (14, 5), (5, 5)][type_]


# ---------------------------------------------------------------- one pass
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("forces", "md"):
        out = []
        if kind == "md":
            s["ctx"].clear_guess()   # a new trajectory: the first step starts from SAD
        for X in s["X"]:
            E = torch.empty(X.shape[0], dtype=torch.float64, device="cuda")
            G = torch.empty_like(X)
            native.pimd_bo_forces_dev(s["ctx"], s["basis"], s["Z"], X, E, G, s["opts"],
                                      torch.cuda.current_stream().cuda_stream)
            out += [E, G]
        return out
    if kind == "images":
        E = torch.empty(len(s["nat"]), dtype=torch.float64, device="cuda")
        G = torch.empty_like(s["X"])
        native.string_images_forces_dev(s["ctx"], s["basis"], s["nat"], s["Z"], s["X"], E, G, s["opts"],
                                        torch.cuda.current_stream().cuda_stream)
        return [E, G]
    if kind == "fock":
        G = torch.empty_like(s["D"])
        native.pimd_fock_dev(s["ctx"], s["basis"], s["Z"], s["X"], s["D"], G, 1e-12, case["fp32_tau"])
        return [G]
    if kind == "eigh":
        V = torch.empty_like(s["A"])
        w = torch.empty(case["nmat"], case["n"], dtype=torch.float64, device="cuda")
        native.pimd_eigh_dev(s["ctx"], s["A"], V, w)
        return [w, V]
    loss, _, grads = s["model"].mlp_grad(case["type"], s["X"], s["Y"])
    return [loss, grads]


# ---------------------------------------------------------------- work
def _quartets(Z, X, kind):
    """Contracted shell quartets with two non-negligible charge distributions
    (an estimate: pairs whose most diffuse primitives overlap, over the
    canonical pairs of pairs whose product is not negligible)."""
    bas = inputs.basis_set(kind)
    sh = [(a, min(s.exps)) for a, z in enumerate(Z) for s in bas[int(z)]]
    at = np.array([a for a, _ in sh])
    ex = np.array([e for _, e in sh])
    d2 = ((X[at][:, None, :] - X[at][None, :, :]) ** 2).sum(-1)
    q = np.exp(-ex[:, None] * ex[None, :] / (ex[:, None] + ex[None, :]) * d2)
    q = np.sort(q[np.triu_indices(len(at))])
    n = np.searchsorted(q, 1e-12 / np.maximum(q, 1e-100), side="left")
    return float((len(q) - n).sum() + len(q)) / 2.0


def work(case):
    kind = case["kind"]
    if kind == "eigh":
        n, m = case["n"], case["nmat"]
        return {"bytes": 8.0 * m * (2 * n * n + n), "flops": 9.0 * m * n ** 3}   # tridiagonal form and back
    if kind == "train":
        na, nb = _head(case["type"])
        dims = 96 * 256 + 2 * 256 * 256 + 256 * na * nb
        return {"bytes": 4.0 * (case["rows"] * (96 + na * nb) + 2 * dims), "flops": 6.0 * case["rows"] * dims}
    # operations per contracted quartet of a Fock build and of the gradient
    # (recursion, set-up and Boys over the primitive quartets that matter)
    fq, gq = (5.7e3, 3.3e4) if case["basis"] == "split_spd" else (1.0e3, 4.0e3)
    if kind == "images":
        mols = [_molecule("water", 1 + i % case["nmax"], i) for i in range(case["images"])]
        calls, iters = 1, 16
    elif kind == "fock":
        mols = [_molecule(case["system"], case["size"], 0)] * case["beads"]
        calls, iters = 1, 1
    else:
        mols = [_molecule("water", case["nwater"], 0)] * case["beads"]
        calls, iters = case.get("steps", 1), 16
    cost, size = {}, 0.0
    flops = 0.0
    for Z, xyz in mols:
        key = (len(Z), float(xyz.sum()))
        if key not in cost:
            cost[key] = _quartets(Z, xyz * inputs.ANGSTROM_TO_BOHR, case["basis"])
        flops += calls * cost[key] * (iters * fq + (gq if kind != "fock" else 0.0))
        n = inputs.nbf_of(inputs.basis_set(case["basis"]), Z)
        size += 16.0 * n * n if kind == "fock" else 8.0 * calls * (6 * len(Z) + 1)
    return {"bytes": size, "flops": flops}


# ---------------------------------------------------------------- exact values
def exact(case, seed):
    if case["kind"] == "eigh":
        A = torch.tensor(_symmetric(case["nmat"], case["n"], seed), device="cuda")
        return [torch.linalg.eigvalsh(A), None]   # the vectors' signs are free
    if case["kind"] == "fock" and case["system"] == "water" and case["size"] <= 2:
        Z, X = _beads("water", case["size"], case["beads"], seed).stacked()
        rng = np.random.default_rng(seed)
        D = [_density(Z, x, case["basis"], rng) for x in X]
        # one replica's matrix costs seconds: the small batches only
        if case["beads"] * case["size"] ** 3 > 16:
            return None
        return [torch.stack([_exact_fock(Z, x, d, case["basis"]) for x, d in zip(X, D)])]
    return None


def _cartesian_functions(Z, X, kind):
    """Primitive Cartesian Gaussians x^l y^m z^n exp(-a r^2) of the basis and
    the matrix [spherical contracted, primitive Cartesian] of coefficients."""
    bas = inputs.basis_set(kind)
    prim, rows = [], []   # (centre, a, (l, m, n))
    s3 = math.sqrt(3.0)
    sph = {0: [[1.0]], 1: np.eye(3).tolist(),
           2: [[0, s3, 0, 0, 0, 0], [0, 0, 0, 0, s3, 0], [-.5, 0, 0, -.5, 0, 1], [0, 0, s3, 0, 0, 0],
               [.5 * s3, 0, 0, -.5 * s3, 0, 0]]}
    comps = {0: [(0, 0, 0)], 1: [(1, 0, 0), (0, 1, 0), (0, 0, 1)],
             2: [(2, 0, 0), (1, 1, 0), (1, 0, 1), (0, 2, 0), (0, 1, 1), (0, 0, 2)]}
    df = {0: 1.0, 1: 1.0, 2: 3.0}
    for z, x in zip(Z, X):
        for sh in bas[int(z)]:
            a = np.array(sh.exps)
            c = np.array(sh.coefs) * (2 * a / math.pi) ** 0.75 * (4 * a) ** (0.5 * sh.l) / math.sqrt(df[sh.l])
            p = a[:, None] + a[None, :]
            c = c / math.sqrt((c[:, None] * c[None, :] * (math.pi / p) ** 1.5 * df[sh.l] / (2 * p) ** sh.l).sum())
            first = len(prim)
            for ai in a:
                prim += [(x, ai, lmn) for lmn in comps[sh.l]]
            nc = len(comps[sh.l])
            for row in sph[sh.l]:
                rows.append([(first + i * nc + k, c[i] * row[k]) for i in range(len(a)) for k in range(nc)])
    M = np.zeros((len(rows), len(prim)))
    for r, items in enumerate(rows):
        for k, v in items:
            M[r, k] = v
    return prim, M


def _exact_fock(Z, X, D, kind):
    """G = J - K/2 with every integral evaluated by quadrature:
    (ab|cd) = 2 pi^{5/2} / (p q sqrt(p + q)) K_ab K_cd int_0^1 Ix Iy Iz e^{-T t^2} dt,
    Ix(t) the two-dimensional integrals of Rys, Dupuis and King; 48
    Gauss-Legendre points on [0, min(1, 6.6 / sqrt T)]."""
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    prim, M = _cartesian_functions(Z, X, kind)
    n = len(prim)
    R = torch.tensor(np.array([p[0] for p in prim]), device=dev)
    e = torch.tensor([p[1] for p in prim], dtype=torch.float64, device=dev)
    l = torch.tensor([p[2] for p in prim], device=dev)
    Mt = torch.tensor(M, device=dev)
    D = torch.tensor(np.asarray(D), device=dev)
    i, j = torch.triu_indices(n, n, device=dev)
    p = e[i] + e[j]
    P = (e[i, None] * R[i] + e[j, None] * R[j]) / p[:, None]
    K = torch.exp(-e[i] * e[j] / p * ((R[i] - R[j]) ** 2).sum(1))
    # (a b| as a sum over the powers (x - A)^k of one centre: the second
    # centre's power expanded about A, coefficients T[pair, axis, k]
    T = torch.zeros(len(i), 3, 5, dtype=torch.float64, device=dev)
    AB = R[i] - R[j]
    for k in range(3):
        mask = l[j] >= k
        binom = torch.where(l[j] == 2, torch.tensor([1, 2, 1], device=dev)[k], 1)
        term = torch.where(mask, binom * AB ** (l[j] - k).clamp(min=0), torch.zeros_like(AB))
        T.scatter_add_(2, (l[i] + k).clamp(max=4).unsqueeze(2), term.unsqueeze(2))
    x, w = np.polynomial.legendre.leggauss(48)
    x = torch.tensor(0.5 * (x + 1.0), device=dev)
    w = torch.tensor(0.5 * w, device=dev)
    # densities of the primitive pairs and contraction: G_sph = M G_prim M^T
    Dp = Mt.T @ D @ Mt
    J = torch.zeros(n, n, dtype=torch.float64, device=dev)
    Kx = torch.zeros(n, n, dtype=torch.float64, device=dev)
    both = torch.where(i == j, 1.0, 2.0)
    Dij = Dp[i, j] * both
    step = max(1, 4_000_000 // (len(i)))
    for b0 in range(0, len(i), step):
        b = slice(b0, min(b0 + step, len(i)))
        pb, q = p[b, None], p[None, :]
        rho = pb * q / (pb + q)
        PQ = P[b, None, :] - P[None, :, :]
        Tq = rho * (PQ ** 2).sum(-1)
        top = (6.6 / Tq.clamp(min=1e-30).sqrt()).clamp(max=1.0)
        pre = 2 * math.pi ** 2.5 / (pb * q * (pb + q).sqrt()) * K[b, None] * K[None, :]
        V = torch.zeros_like(Tq)
        for xk, wk in zip(x, w):
            u2 = (top * xk) ** 2
            f = wk * top * torch.exp(-Tq * u2)
            for ax in range(3):
                f = f * _two_dim(T[b, ax], T[:, ax], P[b, ax] - R[i[b], ax], P[:, ax] - R[i, ax], PQ[..., ax], pb, q,
                                 rho * u2)
            V += f
        V *= pre
        J[i[b], j[b]] = V @ Dij
        # exchange: K_ac += (ab|cd) D_bd over the ordered pairs of both sides
        ib, jb = i[b], j[b]
        for (a1, b1, s1) in ((ib, jb, None), (jb, ib, ib != jb)):
            V1 = V if s1 is None else V * s1[:, None]
            for (c1, d1, s2) in ((i, j, None), (j, i, i != j)):
                W = (V1 if s2 is None else V1 * s2[None, :]) * Dp[b1][:, d1]
                rows = torch.zeros(W.shape[0], n, dtype=torch.float64, device=dev).index_add_(1, c1, W)
                Kx.index_add_(0, a1, rows)
    J = J + J.T - torch.diag(torch.diagonal(J))
    return Mt @ (J - 0.5 * Kx) @ Mt.T


def _two_dim(Tb, Tk, PA, QC, PQ, p, q, ru):
    """sum_{n,m} Tb[n] Tk[m] I(n, m) of one axis, I by the recursion over the
    bra power n and the ket power m at rho t^2 = ru."""
    b00 = ru / (2 * p * q)
    b10 = (1 - ru / p) / (2 * p)
    b01 = (1 - ru / q) / (2 * q)
    c00 = PA[:, None] - ru / p * PQ
    d00 = QC[None, :] + ru / q * PQ
    nb = int(torch.nonzero(Tb.abs().sum(0)).max()) if Tb.numel() else 0
    nk = int(torch.nonzero(Tk.abs().sum(0)).max()) if Tk.numel() else 0
    I = [[None] * (nk + 1) for _ in range(nb + 1)]
    out = 0.0
    for m in range(nk + 1):
        for k in range(nb + 1):
            if m == 0:
                v = torch.ones_like(ru) if k == 0 else c00 * I[k - 1][0]
                if k > 1:
                    v = v + (k - 1) * b10 * I[k - 2][0]
            else:
                v = d00 * I[k][m - 1]
                if m > 1:
                    v = v + (m - 1) * b01 * I[k][m - 2]
                if k > 0:
                    v = v + k * b00 * I[k - 1][m - 1]
            I[k][m] = v
            out = out + Tb[:, k, None] * Tk[None, :, m] * v
    return out
