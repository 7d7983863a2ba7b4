"""The symmetric CUDA-core stage against the FP64 oracle where its plan
changes: meshes below one tile, with a partial last tile, small enough to
share a row's point groups among threads and large enough not to; rules of
V4 symmetry (compact), Z2 symmetry (default) and none (the default rule with
its vertices rotated, which takes the dense stage); kappa = 1 and 2; two
excitations.  Bound on the relative L2 error of the stage increment: 1e-12
(FP64), 1e-5 (FP32), the bounds of the other one-stage tests."""
import numpy as np
import pytest

from oracle import lserk
from oracle.adjoint import gradient
from oracle.refelem import stroud_rule
from synthetic import Dipole, PmlProfile, compact_rule, cube_tet_mesh
from tests.parity_util import (increment_err, make_pair, random_states, rel_err, round_states,
                               to_lib)

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 1e-5}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2006_02551_gb300 import build
    build.build()


def volume_rule(kind, N):
    if kind == "compact":
        return compact_rule(N)
    if kind == "default":
        return None
    r, s, t, w = stroud_rule(N + 1)   # vertices 0 -> 1 -> 2 -> 3 -> 0
    return np.stack([-1.0 - (1 + r + s + t), r, s, w], axis=1)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("N,n_hex,kind,kappa", [
    (1, 1, "compact", 1.0), (1, 10, "default", 1.0), (2, 2, "compact", 2.0),
    (2, 9, "compact", 1.0), (3, 1, "default", 1.0), (3, 8, "default", 2.0),
    (3, 8, "compact", 1.0), (3, 3, "rotated", 1.0), (4, 1, "compact", 1.0),
    (4, 5, "default", 1.0), (4, 7, "compact", 2.0), (4, 8, "compact", 1.0),
    (5, 1, "default", 1.0), (5, 3, "default", 2.0), (5, 3, "compact", 1.0),
    (2, 2, "rotated", 2.0)])
def test_one_stage(N, n_hex, kind, kappa, prec):
    prof = PmlProfile(u0=0.4, L=0.6, sigma_max=20.0, p_sigma=3.0, kappa_max=kappa, eps0=1.5)
    src = tuple(Dipole(x=(0.1, -0.05, 0.2), dir=(0.0, 0.6, 0.8), t0=0.3, width=0.2, batch=b)
                for b in range(2))
    eps = np.random.default_rng(3).uniform(1.0, 4.0, 6 * n_hex ** 3)
    s, sim, mask = make_pair(N, n_hex, 0.15 if n_hex > 1 else 0.0, 1, prof, prec, sources=src,
                             eps=eps, n_batch=2, volume_rule=volume_rule(kind, N))
    st = round_states(random_states(sim.K, sim.Np, 2, 70 + N, mask), prec)
    q0 = to_lib(st)
    s.set_state(q0, 0.0)
    stage, dt, t = 2, 0.004, 0.27
    s.rk_stage(stage, t, dt)
    q, _ = s.get_state()
    s.close()
    for b in range(2):
        rhs = sim.rhs(st[b], t + lserk.RK_C[stage] * dt, b)
        for f in st[b]:
            st[b][f] = st[b][f] + lserk.RK_B[stage] * dt * rhs[f]
    err = increment_err(q, st, q0, mask)
    assert err < TOL[prec], err


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("N,n_hex,kind,kappa,nb", [
    (1, 4, "compact", 1.0, 2), (2, 3, "default", 2.0, 1), (2, 10, "compact", 1.0, 2),
    (3, 2, "rotated", 1.0, 1), (3, 6, "default", 1.0, 1), (4, 3, "compact", 2.0, 1),
    (4, 9, "compact", 1.0, 1), (5, 2, "default", 1.0, 2), (5, 3, "compact", 1.0, 1)])
def test_step_graph(N, n_hex, kind, kappa, nb, prec):
    """Two steps of the step graph: meshes whose classes fit one wave of blocks
    (one launch per stage, the next one's set-up overlapping it), at the edge
    of it and beyond; rules without symmetry.  The state moves by less than
    itself in two steps, so the stage bounds hold for it too."""
    prof = PmlProfile(u0=0.4, L=0.6, sigma_max=20.0, p_sigma=3.0, kappa_max=kappa, eps0=1.5)
    src = tuple(Dipole(x=(0.1, -0.05, 0.2), dir=(0.0, 0.6, 0.8), t0=0.01, width=0.02, batch=b)
                for b in range(nb))
    s, sim, mask = make_pair(N, n_hex, 0.15, 1, prof, prec, sources=src, n_batch=nb,
                             volume_rule=volume_rule(kind, N))
    st = round_states(random_states(sim.K, sim.Np, nb, 80 + N, mask), prec)
    dt = 0.2 * sim.stable_dt(1.0)
    s.set_state(to_lib(st), 0.0)
    s.run_steps(2, dt)
    q, _ = s.get_state()
    s.close()
    st, _, _, _ = sim.run(st, 2, dt)
    assert rel_err(q, st, mask) < TOL[prec]


@pytest.mark.parametrize("N,n_hex,kind", [
    (1, 4, "default"), (2, 1, "compact"), (2, 5, "compact"), (3, 2, "rotated"),
    (3, 3, "default"), (4, 3, "compact"), (4, 2, "default"), (5, 2, "compact"),
    (5, 2, "default")])
def test_fp32_adjoint(N, n_hex, kind):
    """The FP32 reverse stage against the oracle's derivative at partial and
    several tiles, two excitations, the three symmetries of a rule and the
    dense fallback; bound: the 2e-4 of the other FP32 adjoint test."""
    prof = PmlProfile(u0=0.2, L=0.8, sigma_max=20.0, p_sigma=2.0)
    v, e = cube_tet_mesh(n_hex, 0.15 if n_hex > 1 else 0.0, 2)
    eps = np.random.default_rng(3).uniform(1, 4, e.shape[0])
    dirs = ((0.0, 0.6, 0.8), (1.0, 0.0, 0.0))
    src = [Dipole(x=(0.1, 0.05, -0.1), dir=d, t0=0.1, width=0.1, batch=b)
           for b, d in enumerate(dirs)]
    s, sim, _ = make_pair(N, 0, 0.0, 0, prof, "fp32", sources=src, eps=eps, n_batch=2,
                          probes=[(0.3, 0.2, 0.1), (-0.4, 0.3, 0.2)], mesh=(v, e),
                          volume_rule=volume_rule(kind, N))
    dt = 0.5 * sim.stable_dt(1.0)
    s.set_state(None, 0.0)
    J, gE, gS, gP = s.adjoint(8, dt, ckpt_every=3)
    s.close()
    for b in range(2):
        rJ, rE, rS, rP = gradient(sim, eps, prof.sigma_max, prof.p_sigma, 8, dt, batch=b)
        errs = (abs(J[b] - rJ) / abs(rJ), np.linalg.norm(gE[b] - rE) / np.linalg.norm(rE),
                abs(gS[b].sum() - rS) / abs(rS), abs(gP[b].sum() - rP) / abs(rP))
        assert max(errs) < 2e-4, (b, errs)
