"""Host-side checks of the generated recursions (no GPU): the packed
float-float recursion (two mirror-image nodes per operation) must accumulate
what the scalar recursion does, for every class and every accumulator, and the
nuclear-attraction recursion must obey the symmetry of its two shells. The
generated statements are evaluated as they stand."""
import os
import re
import sys

import numpy as np
import pytest

sys.path.insert(0, os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                                "paper_1601_02713_gb300", "csrc"))
import gen_eri as g  # noqa: E402


def _body(code, name):
    """Statements of the generated function `name`, declarations stripped."""
    text = code[code.index(f" {name}("):]
    text = text[text.index("\n{") + 2:text.index("\n}")]
    return [re.sub(r"^const (R|double|dfloat2?) ", "", s.strip()) for s in text.split(";") if s.strip()]


def _fma(a, b, c):
    return a * b + c


@pytest.mark.parametrize("c", g.classes(), ids=g.cls_name)
def test_packed_recursion_equals_scalar(c):
    la, lb, lc, ld = c
    L = sum(c)
    sets = [("acc", la, la + lb, lc, lc + ld, None)]
    n = g.n_range(la, la + lb) * g.n_range(lc, lc + ld)
    rng = np.random.default_rng(sum(x * 7 ** i for i, x in enumerate(c)))
    vec = {v: rng.uniform(-1.0, 1.0, 3) for v in ("PA", "WP", "QC", "WQ")}
    co = {k: rng.uniform(0.5, 1.5) for k in ("o2p", "o2pr", "o2q", "o2qr", "o2pq")}
    F = rng.uniform(0.5, 1.5, L + 1)
    start = rng.normal(size=n)
    # scalar
    env = {f"{v}{i}": vec[v][i] for v in vec for i in range(3)}
    env.update(co, fma=_fma, R=float, Fm=F, acc=start.copy())
    code, _, _ = g.gen_vrr("vrr", L, sets)
    for s in _body(code, "vrr"):
        exec(s, env)
    # packed: a dfloat2 is an array of its two lanes
    code, npk = g.gen_vrr_packed("vrr2", sets)
    unpack = [re.sub(r"\.lane([01])\(\)", r"[\1]", s) for s in _body(code, "vrr2_unpack")]
    acc2 = np.zeros((npk["acc"], 2))
    pk = dict(fma=_fma, exchange=lambda a: a[::-1], acc2=acc2, acc=np.zeros(n))
    for s in unpack:   # start values through the inverse of the unpacking
        dst, src, lane = map(int, re.match(r"acc\[(\d+)\] = acc2\[(\d+)\]\[(\d)\]", s).groups())
        acc2[src, lane] = start[dst]
    # a node that is its own mirror image keeps both lanes equal
    used = {}
    for s in unpack:
        src, lane = re.search(r"acc2\[(\d+)\]\[(\d)\]", s).groups()
        used.setdefault(int(src), set()).add(int(lane))
    for i, lanes in used.items():
        if lanes == {0}:
            acc2[i, 1] = acc2[i, 0]
    for m in range(L + 1):
        pk[f"F{m}"] = np.array([F[m], F[m]])
    for v in vec:
        pk[v + "01"] = np.array([vec[v][0], vec[v][1]])
        pk[v + "2"] = np.array([vec[v][2], vec[v][2]])
    neg = {"no2pr": "o2pr", "no2qr": "o2qr"}
    for k in ("o2p", "no2pr", "o2q", "no2qr", "o2pq"):
        x = -co[neg[k]] if k in neg else co[k]
        for m in range(1, 6):
            pk[k if m == 1 else f"{k}_{m}"] = np.array([m * x, m * x])
    for s in _body(code, "vrr2"):
        if re.match(r"(v|x)\d+ =|acc2\[", s):
            exec(s, pk)
    for s in unpack:
        exec(s, pk)
    scale = np.abs(env["acc"]).max()
    np.testing.assert_allclose(pk["acc"], env["acc"], rtol=0, atol=1e-13 * scale * max(1, L))


@pytest.mark.parametrize("la", range(3))
@pytest.mark.parametrize("lb", range(3))
def test_nuclear_recursion_symmetry(la, lb):
    """(a|b) of shells (la, lb) with P - A, P - B is (b|a) of (lb, la) with the
    two exchanged, for F_m of the form of the Boys function's moments."""
    rng = np.random.default_rng(3 * la + lb)
    PA, PB, PC, o2p = rng.uniform(-1, 1, 3), rng.uniform(-1, 1, 3), rng.uniform(-1, 1, 3), 0.4
    # the recursion is symmetric for the integrals of a Gaussian average over C
    # displacements: F_m = sum_k w_k t_k^m of any nodes, here two
    w, t = rng.uniform(0.5, 1.5, 2), rng.uniform(0.1, 0.9, 2)
    F = np.array([(w * t ** m).sum() for m in range(la + lb + 1)])

    def run(l1, l2, p1, p2):
        env = dict(F=F, PA=p1, PB=p2, PC=PC, o2p=o2p, out=np.zeros(g.ncart(l1) * g.ncart(l2)))
        for s in _body(g.gen_nuclear(l1, l2), f"nuc_{l1}{l2}"):
            exec(s, env)
        return env["out"].reshape(g.ncart(l1), g.ncart(l2))

    np.testing.assert_allclose(run(la, lb, PA, PB), run(lb, la, PB, PA).T, rtol=0, atol=1e-13)
