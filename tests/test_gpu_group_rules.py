"""FP32 groups whose members the grouped variant kernels would serve but for
their volume rules: members of one order with different (N+1)^3-point rules, and
with a rule of no symmetry.  Such a group accepts per_item = 0, launches every
item on its own, says so, and gives each member its own run's values bit for
bit; once the rules agree again the variant kernels run."""
import numpy as np
import pytest

from oracle.refelem import stroud_rule
from synthetic import PmlProfile, cube_tet_mesh

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2006_02551_gb300 import build
    build.build()


def rotated(N):
    r, s, t, w = stroud_rule(N + 1)   # vertices 0 -> 1 -> 2 -> 3 -> 0: no symmetry
    return np.stack([-1.0 - (1 + r + s + t), r, s, w], axis=1)


def swapped(N):
    r, s, t, w = stroud_rule(N + 1)   # vertices 2 <-> 3: the same symmetry, another rule
    return np.stack([r, t, s, w], axis=1)


def member(N, n_hex, rule):
    from paper_2006_02551_gb300 import Solver
    v, e = cube_tet_mesh(n_hex, 0.15, N)
    s = Solver(N, "fp32")
    if rule is not None:
        s.set_quadrature(rule)
    s.set_mesh(v, e)
    s.set_pml(PmlProfile(u0=0.5, L=0.5, sigma_max=20.0, p_sigma=3.0))
    q0 = np.random.default_rng(n_hex).normal(size=s.state_shape())
    return s, q0


@pytest.mark.parametrize("rule", [rotated, swapped])
def test_rules_that_differ_run_per_item(rule):
    from paper_2006_02551_gb300 import Group
    spec = [(2, 4, None), (2, 3, rule(2)), (3, 3, None)]
    pairs = [member(*m) for m in spec]
    members = [p[0] for p in pairs]
    dts = [s.stable_dt(0.5) for s in members]
    ref = []
    for (s, q), dt in zip(pairs, dts):
        s.set_state(q, 0.0)
        s.run_steps(3, dt)
        ref.append(s.get_state()[0])
    g = Group(members)
    g.set_tuning(per_item=False)
    assert g.info()["per_item"]
    g.autotune(dts, reps=5)
    assert g.info()["per_item"]
    for s, q in pairs:
        s.set_state(q, 0.0)
    g.run_steps(3, dts)
    for s, r in zip(members, ref):
        assert np.array_equal(s.get_state()[0], r)
    members[1].set_quadrature(None)
    g.set_tuning(per_item=False)
    assert not g.info()["per_item"]
    for s, q in pairs:
        s.set_state(q, 0.0)
    g.run_steps(3, dts)
    assert np.array_equal(members[0].get_state()[0], ref[0])
    g.close()
    for s in members:
        s.close()
