"""Sources by the hundred in one tile of elements: nine dipoles of every
excitation in each element of a block of the mesh, listed in an order that
follows neither the elements nor the excitations.  One stage on every stage
kernel, and the gradient, against the FP64 oracle; bounds as in the other
one-stage and adjoint tests."""
import numpy as np
import pytest

from oracle import lserk
from oracle.adjoint import gradient
from oracle.refelem import stroud_rule
from synthetic import Dipole, PmlProfile, compact_rule, cube_tet_mesh
from tests.parity_util import increment_err, make_pair, random_states, round_states, to_lib

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 1e-5, "tf32": 1e-2, "bf16": 3e-2}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2006_02551_gb300 import build
    build.build()


def many(v, e, per, nb, seed):
    """per dipoles of each excitation in every element of (0, 0.6)^3, shuffled."""
    rng = np.random.default_rng(seed)
    c = v[e].mean(axis=1)
    out = []
    for k in np.nonzero(((c > 0) & (c < 0.6)).all(axis=1))[0]:
        for b in range(nb):
            for _ in range(per):
                x = rng.dirichlet(np.full(4, 3.0)) @ v[e[k]]
                d = rng.normal(size=3)
                out.append(Dipole(x=tuple(x), dir=tuple(d / np.linalg.norm(d)), t0=0.3, width=0.2,
                                  batch=b))
    return [out[i] for i in rng.permutation(len(out))]


@pytest.mark.parametrize("prec,N,kind,pml", [
    ("fp64", 4, "compact", True), ("fp64", 4, "compact", False), ("fp64", 2, "rotated", True),
    ("fp32", 4, "compact", True), ("fp32", 2, "default", False), ("fp32", 3, "rotated", True),
    ("tf32", 3, "compact", True), ("tf32", 3, "default", True), ("bf16", 2, "default", False)])
def test_one_stage(prec, N, kind, pml):
    v, e = cube_tet_mesh(10, 0.1, 3)
    # every element in the PML class, or none
    prof = PmlProfile(u0=0.0 if pml else 5.0, L=1.0, sigma_max=20.0, p_sigma=3.0)
    if kind == "rotated":   # no symmetry: the dense stage
        r, s_, t, w = stroud_rule(N + 1)
        rule = np.stack([-1.0 - (1 + r + s_ + t), r, s_, w], axis=1)
    else:
        rule = compact_rule(N) if kind == "compact" else None
    src = many(v, e, 9, 2, 5)
    s, sim, mask = make_pair(N, 0, 0.0, 0, prof, prec, sources=src, n_batch=2, mesh=(v, e),
                             volume_rule=rule)
    assert mask.all() if pml else not mask.any()
    st = round_states(random_states(sim.K, sim.Np, 2, 40 + N, mask), prec)
    q0 = to_lib(st)
    s.set_state(q0, 0.0)
    stage, dt, t = 1, 0.004, 0.1
    s.rk_stage(stage, t, dt)
    q, _ = s.get_state()
    s.close()
    for b in range(2):
        rhs = sim.rhs(st[b], t + lserk.RK_C[stage] * dt, b)
        for f in st[b]:
            st[b][f] = st[b][f] + lserk.RK_B[stage] * dt * rhs[f]
    err = increment_err(q, st, q0, mask)
    assert err < TOL[prec], err


@pytest.mark.parametrize("prec,tol,kind", [("fp64", 1e-10, "compact"), ("fp32", 2e-4, "compact"),
                                           ("fp32", 2e-4, "rotated")])
def test_gradient(prec, tol, kind):
    N = 2
    v, e = cube_tet_mesh(10, 0.1, 3)
    prof = PmlProfile(u0=0.0, L=1.0, sigma_max=10.0, p_sigma=2.0)
    if kind == "rotated":
        r, s_, t, w = stroud_rule(N + 1)
        rule = np.stack([-1.0 - (1 + r + s_ + t), r, s_, w], axis=1)
    else:
        rule = compact_rule(N)
    eps = np.random.default_rng(3).uniform(1, 4, e.shape[0])
    src = many(v, e, 9, 1, 6)
    s, sim, _ = make_pair(N, 0, 0.0, 0, prof, prec, sources=src, eps=eps,
                          probes=[(0.3, 0.2, 0.1), (-0.4, 0.3, 0.2)], mesh=(v, e), volume_rule=rule)
    dt = 0.5 * sim.stable_dt(1.0)
    s.set_state(None, 0.0)
    J, gE, gS, gP = s.adjoint(3, dt, ckpt_every=2)
    s.close()
    rJ, rE, rS, rP = gradient(sim, eps, prof.sigma_max, prof.p_sigma, 3, dt)
    errs = (abs(J[0] - rJ) / abs(rJ), np.linalg.norm(gE[0] - rE) / np.linalg.norm(rE),
            abs(gS[0].sum() - rS) / abs(rS), abs(gP[0].sum() - rP) / abs(rP))
    assert max(errs) < tol, errs
