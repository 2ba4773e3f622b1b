"""Error of the float-float kernels on the GPU beside FP64's, for a Fock matrix
and a two-electron gradient at one fixed density.

An element that the molecule does not hold, with an exponent outside the range
of the float-float kernels, forces FP64. Tolerance: a float-float operation
leaves a few 2^-48 of its largest term, so the rounding of a sum stays below
2^-46 of its norm. The Fock matrix is compared with an unscreened FP64 build's:
the cutoffs may leave what they leave in FP64. The gradient kernels' cutoffs are
the FP64 kernels', so there the two are compared with each other."""
import numpy as np
import pytest

from paper_1601_02713_gb300 import inputs, native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROUNDING = 2.0 ** -46


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return native.Context(0)


def _bases(kind):
    bas = inputs.basis_set(kind)
    return native.Basis(bas), native.Basis({**bas, 2: [inputs.Shell(0, [1e9], [1.0])]})


def _fock(ctx, B, Z, X, D, tau=1e-12):
    Dt = torch.tensor(D, device="cuda")
    G = torch.zeros_like(Dt)
    native.pimd_fock_dev(ctx, B, Z, X, Dt, G, tau)
    return G.cpu().numpy()


def _density(ctx, B, Z, X):
    """A few damped Roothaan steps from the core Hamiltonian."""
    out = []
    for x in X:
        S, T, V = native.pimd_one_electron(ctx, B, Z, x)[:3]
        w, U = np.linalg.eigh(S)
        L = U / np.sqrt(w)
        F, D = T + V, None
        for _ in range(5):
            C = L @ np.linalg.eigh(L.T @ F @ L)[1][:, :int(Z.sum()) // 2]
            D = 2.0 * C @ C.T if D is None else C @ C.T + 0.5 * D
            F = T + V + _fock(ctx, B, Z, x[None], D[None])[0]
        out.append(D)
    return np.array(out)


class _Device:
    def __init__(self, ptr, n):
        self.__cuda_array_interface__ = dict(shape=(n,), typestr="<f8", data=(ptr, False), version=3)


def _gradient(ctx, B, Z, X, G, parts=4, first=1):
    """Two-electron gradient at the density of the Fock matrix h + G: one SCF
    iteration of the force-parallel split, whose reduction puts G in the place
    of the sum; the shares of all processes but the first, which adds the
    one-electron part (first = 0: with it). The tiles are dealt out the same way
    in every call."""
    half = torch.tensor(0.5 * G, device="cuda").reshape(-1)
    out = []

    def reduce(ptr, n):
        v = torch.as_tensor(_Device(ptr, n), device="cuda")
        if n == half.numel():
            v.copy_(half)
            torch.cuda.synchronize()
        else:
            out.append(v.cpu().numpy().copy())

    for rank in range(first, parts):
        native.pimd_bo_forces(ctx, B, Z, X, native.scf_opts(guess=0, max_iter=1, split_size=parts, split_rank=rank,
                                                            reduce=reduce), check=False)
    return np.sum(out, axis=0)


def _check(ctx, kind, Z, X):
    B, W = _bases(kind)
    D = _density(ctx, W, Z, X)
    ref = _fock(ctx, W, Z, X, D, 0.0)
    df, fp64 = [np.linalg.norm(_fock(ctx, b, Z, X, D) - ref) / np.linalg.norm(ref) for b in (B, W)]
    assert df < fp64 + ROUNDING
    df, fp64 = [_gradient(ctx, b, Z, X, ref) for b in (B, W)]
    assert np.linalg.norm(df - fp64) < ROUNDING * np.linalg.norm(fp64)


@pytest.mark.parametrize("offset", [0.0, 100.0, 9000.0])
def test_no_further_from_exact_than_fp64_at_any_offset(ctx, offset):
    """Every class of the s/p/d basis, with the molecule at the origin and up to
    the largest coordinates that the float-float kernels take."""
    Z, X = inputs.beads(*inputs.water_dimer_geometry(5), 1, 77).stacked()
    X = np.ascontiguousarray(X + offset * np.array([1.0, -0.7, 0.3]))
    _check(ctx, "split_spd", Z, X)


@pytest.mark.parametrize("kind,nwater", [("min_sp", 1), ("min_sp", 3), ("split_spd", 1), ("split_spd", 4)])
def test_no_further_from_exact_than_fp64(ctx, kind, nwater):
    """Both bases, from a molecule of which the cutoffs drop nothing to one of
    which they drop most."""
    Z, X = inputs.beads(*inputs.water_cluster_geometry(nwater, 2), 1, 31).stacked()
    _check(ctx, kind, Z, X)


def test_gradient_rounding_below_that_of_fp64(ctx):
    """The float-float part adds less than half of the distance between two FP64
    gradients (FP64 atomics in another order) at one density: an independent
    error of that size raises the whole by an eighth."""
    Z, X = inputs.beads(*inputs.water_cluster_geometry(8, 2), 1, 2064).stacked()
    B, W = _bases("split_spd")
    ref = _fock(ctx, W, Z, X, _density(ctx, W, Z, X))
    whole = [_gradient(ctx, W, Z, X, ref, first=0) for _ in range(3)]
    spread = np.mean([np.linalg.norm(whole[i] - whole[i - 1]) for i in range(3)])
    df, fp64 = [np.mean([_gradient(ctx, b, Z, X, ref) for _ in range(3)], axis=0) for b in (B, W)]
    assert np.linalg.norm(df - fp64) < 0.5 * spread


@pytest.mark.parametrize("tau,prim,fp64", [(1e-13, 0.2, True), (0.99e-12, 1.0, True), (1e-12, 1.0, False),
                                           (1e-12, 1.0 / 81.0, False), (1e-12, 0.01, True)])
def test_a_tighter_cutoff_of_either_kind_keeps_fp64(ctx, tau, prim, fp64):
    """Launch for launch the calls of the basis that is outside the range."""
    Z, X = inputs.beads(*inputs.water_cluster_geometry(1, 2), 1, 5).stacked()

    def launches(b):
        native.pimd_bo_forces(ctx, b, Z, X, native.scf_opts(guess=0, max_iter=2, schwarz_tau=tau, prim_screen=prim),
                              check=False)
        return native.pimd_last_stats(ctx)["kernel_launches"]   # of the last forces call

    B, W = _bases("split_spd")
    assert (launches(B) == launches(W)) == fp64


@pytest.mark.parametrize("scale", [300.0, 1e6])
def test_large_densities_leave_the_long_classes_to_fp64(ctx, scale):
    """p and d shells of which nothing is screened and a density so large that
    the cutoffs do not matter: what stays in float-floats is below 2^43 times the
    cutoff, and the rounding below the 2^-46 of the norm that a build is allowed."""
    sh = [inputs.Shell(2, [1.3, 0.5], [0.4, 0.7]), inputs.Shell(1, [0.8], [1.0])]
    B, W = native.Basis({1: sh}), native.Basis({1: sh, 2: [inputs.Shell(0, [1e9], [1.0])]})
    Z = np.array([1, 1], np.int32)
    X = np.array([[[0.0, 0.0, 0.0], [0.2, 0.3, 1.6]]])
    D = np.random.default_rng(3).normal(size=(1, B.nbf(Z), B.nbf(Z)))
    D = scale * (D + D.transpose(0, 2, 1))
    ref = _fock(ctx, W, Z, X, D, 0.0)
    df, fp64 = [np.linalg.norm(_fock(ctx, b, Z, X, D) - ref) / np.linalg.norm(ref) for b in (B, W)]
    assert df < fp64 + ROUNDING


@pytest.mark.parametrize("coefs,exps", [([1.0, -0.999], [9e7, 8.9e7]), ([1.0], [9e7])])
def test_large_prefactors_keep_fp64(ctx, coefs, exps):
    """Tight p and d shells whose prefactors' products are outside FP32, with
    coefficients that nearly cancel and without: the basis outside the range by
    its exponents gives the same matrix, up to the order of the FP64 additions
    (2^-46 of the norm)."""
    sh = [inputs.Shell(2, exps, coefs), inputs.Shell(1, exps, coefs), inputs.Shell(0, [1.1], [1.0])]
    B, W = native.Basis({1: sh}), native.Basis({1: sh, 2: [inputs.Shell(0, [1e9], [1.0])]})
    Z = np.array([1, 1], np.int32)
    X = np.array([[[0.0, 0.1, 0.0], [3e-4, -2e-4, 1e-4]]])
    D = np.random.default_rng(4).normal(size=(1, B.nbf(Z), B.nbf(Z))) * 1e-9
    D = D + D.transpose(0, 2, 1)
    g, ref = [_fock(ctx, b, Z, X, D) for b in (B, W)]
    assert np.isfinite(ref).all() and np.isfinite(g).all()
    assert np.linalg.norm(g - ref) < ROUNDING * np.linalg.norm(ref)


@pytest.mark.parametrize("second", [-0.95, -0.7])
def test_contractions_that_cancel_keep_fp64(ctx, second):
    """Shells of two nearly equal primitives with coefficients of opposite sign:
    the contracted integrals are 1e2 to 1e5 times smaller than the primitive ones,
    and no further from exact than in FP64."""
    sh = [inputs.Shell(l, [1.0, 0.9], [1.0, second]) for l in (2, 1, 0)]
    B, W = native.Basis({1: sh}), native.Basis({1: sh, 2: [inputs.Shell(0, [1e9], [1.0])]})
    Z = np.array([1, 1], np.int32)
    X = np.array([[[0.0, 0.1, 0.0], [0.7, -0.5, 2.1]]])
    D = np.random.default_rng(4).normal(size=(1, B.nbf(Z), B.nbf(Z))) * 1e-2
    D = D + D.transpose(0, 2, 1)
    ref = _fock(ctx, W, Z, X, D, 0.0)
    df, fp64 = [np.linalg.norm(_fock(ctx, b, Z, X, D) - ref) / np.linalg.norm(ref) for b in (B, W)]
    assert df < fp64 + ROUNDING


def _profiled(fn):
    """(fn(), kernels that ran on the device meanwhile)"""
    from torch.profiler import ProfilerActivity, profile

    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        out = fn()
        torch.cuda.synchronize()
    return out, sum(1 for e in p.events() if "_kernel" in e.name)


@pytest.mark.parametrize("fp32_tau", [0.0, 1e-15, 1e-6])
def test_launch_counter_counts_what_runs(ctx, fp32_tau):
    """The counter's difference between the float-float and the FP64 form of a
    call is that of the kernels seen by the profiler, in FP64 and mixed
    precision, and for an FP32 bound below the gradient's quartet cutoff (no
    FP32 launch)."""
    Z, X = inputs.beads(*inputs.water_cluster_geometry(1, 2), 1, 5).stacked()

    def launches(b, f):
        native.pimd_bo_forces(ctx, b, Z, X, native.scf_opts(guess=0, max_iter=1, use_graphs=0, fp32_tau=f),
                              check=False)
        return native.pimd_last_stats(ctx)["kernel_launches"]

    B, W = _bases("split_spd")
    launches(B, fp32_tau)
    _profiled(lambda: launches(W, 0.0))   # one-time set-up of the library and of the profiler
    n0, seen0 = _profiled(lambda: launches(W, 0.0))
    n1, seen1 = _profiled(lambda: launches(B, fp32_tau))
    assert seen0 > 40
    assert n1 - n0 == seen1 - seen0
