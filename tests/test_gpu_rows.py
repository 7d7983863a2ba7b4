"""One stage of the row-owned tensor-core kernel on both element classes
against the FP64 oracle where its tiles can go wrong: fewer elements than a
tile, partial last tiles, one or several tiles per block, two excitations, no
PML at all and PML everywhere, both volume rules, materials.  Bounds on the
relative L2 error of the stage increment: 1e-2 (TF32), 3e-2 (BF16), those of
the other one-stage tests of these precisions."""
import numpy as np
import pytest

from oracle import lserk
from synthetic import Dipole, PmlProfile, compact_rule
from tests.parity_util import increment_err, make_pair, random_states, round_states, to_lib

pytestmark = pytest.mark.gpu

TOL = {"tf32": 1e-2, "bf16": 3e-2}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2006_02551_gb300 import build
    build.build()


@pytest.mark.parametrize("prec", ["tf32", "bf16"])
@pytest.mark.parametrize("N,n_hex,u0,compact", [
    (1, 1, None, True), (1, 9, 0.4, True), (2, 2, None, False), (2, 7, 0.4, True),
    (3, 1, 0.4, True), (3, 9, 0.4, False), (4, 1, None, True), (4, 9, 0.4, True),
    (5, 1, None, True), (5, 2, 0.0, True), (5, 7, 0.4, True)])
def test_one_stage_both_classes(N, n_hex, u0, compact, prec):
    prof = None if u0 is None else PmlProfile(u0=u0, L=1.0 - u0, sigma_max=20.0, p_sigma=3.0,
                                              eps0=1.5)
    src = tuple(Dipole(x=(0.1, -0.05, 0.2), dir=(0.0, 0.6, 0.8), t0=0.3, width=0.2, batch=b)
                for b in range(2))
    K = 6 * n_hex ** 3
    rng = np.random.default_rng(3)
    eps, mu = rng.uniform(1.0, 4.0, K), rng.uniform(1.0, 2.0, K)
    s, sim, mask = make_pair(N, n_hex, 0.15 if n_hex > 1 else 0.0, 1, prof, prec, sources=src,
                             eps=eps, mu=mu, n_batch=2,
                             volume_rule=compact_rule(N) if compact else None)
    st = round_states(random_states(sim.K, sim.Np, 2, 90 + N, mask), prec)
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
