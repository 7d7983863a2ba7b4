"""Caller's volume rules of unusual form against the FP64 oracle on the same
rule: points listed more than once (what averaging a rule over the vertex
permutations gives).
Bounds on the relative L2 error of the stage increment: 1e-12 (FP64), 1e-5
(FP32), 1e-2 (TF32), those of the other one-stage tests; on the gradient 1e-10
(FP64), 2e-4 (FP32), those of the other adjoint tests."""
import numpy as np
import pytest

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
