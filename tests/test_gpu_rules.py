"""Caller's volume rules of unusual form against the FP64 oracle on the same
rule: points listed more than once (what averaging a rule over the vertex
permutations gives), and a point on a vertex whose coordinate rounds above 1.
Bounds on the relative L2 error of the stage increment: 1e-12 (FP64), 1e-5
(FP32), 1e-2 (TF32), those of the other one-stage tests; on the gradient 1e-10
(FP64), 2e-4 (FP32), those of the other adjoint tests."""
import itertools
import math

import numpy as np
import pytest
from scipy.special import roots_jacobi

from oracle import lserk
from oracle.adjoint import gradient
from synthetic import Dipole, PmlProfile, compact_rule, cube_tet_mesh
from tests.parity_util import increment_err, make_pair, random_states, round_states, to_lib

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 1e-5, "tf32": 1e-2}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2006_02551_gb300 import build
    build.build()


def one_stage(N, rule, prec, kappa=1.0):
    prof = PmlProfile(u0=0.4, L=0.6, sigma_max=20.0, p_sigma=3.0, kappa_max=kappa)
    s, sim, mask = make_pair(N, 2, 0.15, 1, prof, prec, volume_rule=rule)
    st = round_states(random_states(sim.K, sim.Np, 1, 90 + N, mask), prec)
    q0 = to_lib(st)
    s.set_state(q0, 0.0)
    stage, dt = 1, 0.004
    s.rk_stage(stage, 0.0, dt)
    q, _ = s.get_state()
    s.close()
    rhs = sim.rhs(st[0], lserk.RK_C[stage] * dt, 0)
    for f in st[0]:
        st[0][f] = st[0][f] + lserk.RK_B[stage] * dt * rhs[f]
    return increment_err(q, st, q0, mask)


# ------------------------------------------------------- repeated points

def repeated(N, kind):
    """twice: every point listed twice at half weight, next to each other;
    again: the same, the whole list after itself; split, split_last: one point
    in two halves; uneven: every point as 1/4 and 3/4 of its weight."""
    r = compact_rule(N)
    if kind in ("split", "split_last"):
        q = 0 if kind == "split" else r.shape[0] - 1
        r = np.concatenate([r, r[q:q + 1]])
        r[q, 3] *= 0.5
        r[-1, 3] *= 0.5
        return r
    a, b = r.copy(), r.copy()
    a[:, 3] *= 0.25 if kind == "uneven" else 0.5
    b[:, 3] *= 0.75 if kind == "uneven" else 0.5
    if kind == "again":
        return np.concatenate([a, b])
    return np.stack([a, b], axis=1).reshape(-1, 4)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("N,kind,kappa", [
    (1, "twice", 1.0), (1, "split", 2.0), (2, "split", 1.0), (2, "split_last", 2.0),
    (3, "twice", 1.0), (3, "again", 2.0), (3, "split", 1.0), (4, "twice", 1.0),
    (4, "again", 2.0), (4, "uneven", 1.0), (4, "split", 1.0), (5, "twice", 1.0),
    (5, "split", 1.0)])
def test_repeated_points_one_stage(N, kind, kappa, prec):
    err = one_stage(N, repeated(N, kind), prec, kappa)
    assert err < TOL[prec], err


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("fp32", 2e-4)])
@pytest.mark.parametrize("N,kind", [(4, "twice"), (2, "split")])
def test_repeated_points_gradient(N, kind, prec, tol):
    prof = PmlProfile(u0=0.2, L=0.8, sigma_max=20.0, p_sigma=2.0)
    v, e = cube_tet_mesh(2, 0.15, 2)
    eps = np.random.default_rng(3).uniform(1, 4, e.shape[0])
    src = [Dipole(x=(0.1, 0.05, -0.1), dir=(0.0, 0.6, 0.8), t0=0.1, width=0.1)]
    s, sim, _ = make_pair(N, 0, 0.0, 0, prof, prec, sources=src, eps=eps,
                          probes=[(0.3, 0.2, 0.1), (-0.4, 0.3, 0.2)], mesh=(v, e),
                          volume_rule=repeated(N, kind))
    dt = 0.5 * sim.stable_dt(1.0)
    s.set_state(None, 0.0)
    J, gE, gS, gP = s.adjoint(6, dt, ckpt_every=4)
    s.close()
    rJ, rE, rS, rP = gradient(sim, eps, prof.sigma_max, prof.p_sigma, 6, dt)
    errs = (abs(J[0] - rJ) / abs(rJ), np.linalg.norm(gE[0] - rE) / np.linalg.norm(rE),
            abs(gS[0].sum() - rS) / abs(rS), abs(gP[0].sum() - rP) / abs(rP))
    assert max(errs) < tol, errs


# ------------------------------------------- a point one ulp beyond a vertex

def radau(n, al, right):
    """n-point rule on [-1, 1] for the weight (1 - x)^al with the end point -1
    (right: +1, al = 0) among its points; degree 2n - 2."""
    if right:
        x, w = radau(n, al, False)
        return -x[::-1], w[::-1]
    x, v = roots_jacobi(n - 1, al, 1)     # the weight times (1 + x)
    w = v / (1.0 + x)
    total = 2.0 ** (al + 1) / (al + 1)
    return np.concatenate([[-1.0], x]), np.concatenate([[total - w.sum()], w])


def vertex_rule(N, kind):
    """Rules with a point on vertex 2 of the reference tetrahedron, written
    as r = 1 + 2^-52.  conical: the product of Radau rules ((N + 1)^3 points, no
    symmetry); symmetric (N = 2): 19 points in fully symmetric orbits (vertices,
    two of (a, a, a, 1 - 3a), one of (b, b, 1/2 - b, 1/2 - b), centroid), the
    weights from the moments of degree 4."""
    if kind == "conical":
        (a, wa), (b, wb), (c, wc) = (radau(N + 1, 0, True), radau(N + 1, 1, False),
                                     radau(N + 1, 2, False))
        A, B, C = (t.ravel() for t in np.meshgrid(a, b, c, indexing="ij"))
        s = (1 + B) * (1 - C) / 2 - 1
        rule = np.stack([(1 + A) * (1 - B) * (1 - C) / 4 - 1, s, C,
                         np.einsum("i,j,k->ijk", wa, wb, wc).ravel() / 8], axis=1)
    else:
        orbits = [sorted(set(itertools.permutations(p))) for p in
                  ((1.0, 0.0, 0.0, 0.0), (0.14, 0.14, 0.14, 1 - 3 * 0.14),
                   (0.33, 0.33, 0.33, 1 - 3 * 0.33), (0.06, 0.06, 0.44, 0.44), (0.25,) * 4)]
        exps = [e for e in itertools.product(range(5), repeat=4) if sum(e) == 4]
        A = [[sum(np.prod(np.power(p, e)) for p in o) for o in orbits] for e in exps]
        m = [8.0 * math.prod(math.factorial(k) for k in e) / math.factorial(7) for e in exps]
        w = np.linalg.lstsq(np.array(A), np.array(m), rcond=None)[0]
        assert w.min() > 0
        lam = np.array([p for o in orbits for p in o])
        rule = np.concatenate([2 * lam[:, 1:] - 1,
                               np.concatenate([[x] * len(o) for x, o in zip(w, orbits)])[:, None]], 1)
    q = np.nonzero(np.abs(rule[:, 0] - 1.0) < 1e-12)[0]
    assert q.size == 1
    rule[q[0], :3] = (np.nextafter(1.0, 2.0), -1.0, -1.0)
    return rule


@pytest.mark.parametrize("N,kind,prec,kappa", [
    (2, "symmetric", "fp64", 1.0), (2, "symmetric", "fp32", 2.0), (1, "conical", "fp64", 1.0),
    (3, "conical", "fp64", 2.0), (3, "conical", "fp32", 1.0), (4, "conical", "fp32", 2.0),
    (1, "conical", "tf32", 1.0), (2, "conical", "tf32", 1.0)])
def test_vertex_point_keeps_its_sample(N, kind, prec, kappa):
    err = one_stage(N, vertex_rule(N, kind), prec, kappa)
    assert err < TOL[prec], err
