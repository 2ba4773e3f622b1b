"""Float-float ERI kernels, lane sharing and their limits on the GPU, against
the CPU oracle's Fock matrix of a fixed density.

Tolerance of a Fock element: the integral cutoff leaves 1e-12 times the number
of screened quartets that reach it (a few hundred at these sizes), the
float-float rounding a few 1e-14 of the element's terms (at most some 1e2
hartree): 1e-10 of the largest element covers both."""
import numpy as np
import pytest

import oracle as O
from paper_1601_02713_gb300 import inputs, native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL = 1e-10


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return native.Context(0)


def _density(N, nrep, seed):
    rng = np.random.default_rng(seed)
    D = rng.normal(size=(nrep, N, N)) * 0.3
    return D + D.transpose(0, 2, 1)


def _gpu_tau(ctx, B, Z, Xs, D, tau):
    Dt = torch.tensor(D, device="cuda")
    G = torch.zeros_like(Dt)
    native.pimd_fock_dev(ctx, B, Z, Xs, Dt, G, tau)
    return G.cpu().numpy()


def _gpu(ctx, B, Z, Xs, D):
    return _gpu_tau(ctx, B, Z, Xs, D, 1e-12)


def _check(bas, Z, Xs, D, G, tol=TOL):
    for k in range(len(Xs)):
        ob = O.OracleBasis.build(bas, Z, Xs[k])
        J, K, _ = O.jk(ob, D[k], 1e-12)
        ref = J - 0.5 * K
        err = np.abs(G[k] - ref).max()
        assert err < tol * max(1.0, np.abs(ref).max()), (k, err)


@pytest.mark.parametrize("kind,nrep", [("min_sp", 1), ("min_sp", 7), ("split_spd", 1), ("split_spd", 2)])
def test_small_batches(ctx, kind, nrep):
    """One replica (many lanes to a quartet, several blocks to a tile) and a
    few, both bases: every class of the s/p and s/p/d bases."""
    bas = inputs.basis_set(kind)
    B = native.Basis(bas)
    Z, Xs = inputs.beads(*inputs.water_dimer_geometry(5), nrep, 77).stacked()
    D = _density(B.nbf(Z), nrep, 3)
    _check(bas, Z, Xs, D, _gpu(ctx, B, Z, Xs, D))


def test_boys_switch_points(ctx):
    """Two H atoms at distances that put rho R^2 on both sides of the Boys
    table's end (40) and of the point where e^-T is dropped (72), for exponents
    of both shells, and at R = 0.05."""
    bas = {1: [inputs.Shell(0, [0.7], [1.0]), inputs.Shell(1, [0.7], [1.0]), inputs.Shell(2, [0.7], [1.0])]}
    B = native.Basis(bas)
    Z = np.array([1, 1], np.int32)
    # same-centre pairs: p = q = 1.4, rho = 0.7
    T = [39.9, 39.999999, 40.0, 40.000001, 40.1, 55.3, 71.9, 72.0, 72.1, 200.0]
    R = [0.05] + [np.sqrt(t / 0.7) for t in T]
    Xs = np.zeros((len(R), 2, 3))
    Xs[:, 1] = np.array(R)[:, None] * np.array([0.48, -0.6, 0.64])
    D = _density(B.nbf(Z), len(R), 9)
    _check(bas, Z, Xs, D, _gpu(ctx, B, Z, Xs, D))


@pytest.mark.parametrize("exp", [4e7, 4e8, 3e-7])
def test_extreme_exponents(ctx, exp):
    """A tight shell inside and outside the range of the float-float kernels
    and a diffuse one outside (then every quartet is FP64)."""
    bas = {1: [inputs.Shell(0, [exp], [1.0]), inputs.Shell(0, [1.1, 0.3], [0.5, 0.5]), inputs.Shell(1, [0.8], [1.0])]}
    B = native.Basis(bas)
    Z = np.array([1, 1], np.int32)
    Xs = np.array([[[0.0, 0.1, 0.0], [0.3, -0.2, 1.3]]])
    D = _density(B.nbf(Z), 1, 4)
    _check(bas, Z, Xs, D, _gpu(ctx, B, Z, Xs, D))


def test_far_coordinates(ctx):
    """Coordinates beyond the float-float kernels' range (1e4 bohr): the FP64
    path, equal to the molecule at the origin up to the rounding of the
    coordinates themselves (2e4 bohr: 4e-12, times a derivative of at most 1e2
    hartree per bohr and some 1e2 terms)."""
    bas = inputs.basis_set("split_spd")
    B = native.Basis(bas)
    Z, Xs = inputs.beads(*inputs.water_cluster_geometry(1, 2), 2, 5).stacked()
    D = _density(B.nbf(Z), 2, 6)
    G0 = _gpu(ctx, B, Z, Xs, D)
    G1 = _gpu(ctx, B, Z, Xs + np.array([2.0e4, -3.0e4, 1.5e4]), D)
    np.testing.assert_allclose(G1, G0, rtol=0, atol=1e-7)
    assert not np.array_equal(G1, G0)


@pytest.mark.parametrize("tau,fp64", [(0.0, True), (1e-15, True), (1e-12, False)])
def test_tight_cutoffs_keep_fp64(ctx, tau, fp64):
    """A cutoff below the default asks for less than the float-float rounding:
    the build then takes the FP64 path, launch for launch the one that an element
    outside the float-float range forces (the molecule does not hold it)."""
    bas = inputs.basis_set("split_spd")
    wide = dict(bas)
    wide[2] = [inputs.Shell(0, [1e9], [1.0])]
    Z, Xs = inputs.beads(*inputs.water_cluster_geometry(1, 2), 1, 5).stacked()
    B = native.Basis(bas)
    D = _density(B.nbf(Z), 1, 6)

    def launches(b):
        n0 = native.pimd_last_stats(ctx)["kernel_launches"]
        _gpu_tau(ctx, b, Z, Xs, D, tau)
        return native.pimd_last_stats(ctx)["kernel_launches"] - n0

    assert (launches(B) == launches(native.Basis(wide))) == fp64


@pytest.mark.parametrize("n,nmat", [(1, 3), (2, 1), (31, 2), (64, 5), (65, 1), (127, 2), (129, 1), (193, 1)])
def test_eigensolver_sizes(ctx, n, nmat):
    """The rotations from an FP32 angle over the column lengths, odd sizes,
    degenerate and widely scaled spectra."""
    rng = np.random.default_rng(n)
    A = rng.normal(size=(nmat, n, n))
    A = A + A.transpose(0, 2, 1)
    A[-1] = np.diag(np.repeat(rng.uniform(-1, 1, (n + 3) // 4), 4)[:n]) + 1e-3 * A[-1]   # clusters of four
    if nmat > 1:
        A[0] *= 1e60
    if nmat > 2:
        A[1] *= 1e-9
    At = torch.tensor(A, device="cuda")
    V, w = torch.empty_like(At), torch.empty(nmat, n, dtype=torch.float64, device="cuda")
    native.pimd_eigh_dev(ctx, At, V, w)
    V, w = V.cpu().numpy(), w.cpu().numpy()
    for k in range(nmat):
        # the solver works on A + sigma I with sigma >= 1 - (Gershgorin bound): its scale
        scale = 1.0 + np.abs(A[k]).sum(1).max()
        np.testing.assert_allclose(w[k], np.linalg.eigvalsh(A[k]), rtol=0, atol=1e-13 * scale * max(n, 8))
        np.testing.assert_allclose(V[k].T @ V[k], np.eye(n), rtol=0, atol=1e-12)
        np.testing.assert_allclose((V[k] * w[k]) @ V[k].T, A[k], rtol=0, atol=1e-12 * scale)
