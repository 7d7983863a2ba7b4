"""Failure detection in grouped stepping: a bounded device-side wait that runs
out in a member's launch makes wadg_group_run_steps return WADG_ETIMEOUT and
name the member, the flag does not outlive the call, and the group steps as
before afterwards.  The wait runs out because wadg_arm_wait_timeout makes one
block issue a product without its completion signal; nothing here faults or
waits without a limit."""
import numpy as np
import pytest

from synthetic import PmlProfile, compact_rule, cube_tet_mesh

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2006_02551_gb300 import build
    build.build()


def member(N, n_hex, prec, compact):
    from paper_2006_02551_gb300 import Solver
    v, e = cube_tet_mesh(n_hex, 0.15, N)
    s = Solver(N, prec)
    if compact:
        s.set_quadrature(compact_rule(N))
    s.set_mesh(v, e)
    s.set_pml(PmlProfile(u0=0.5, L=0.5, sigma_max=20.0, p_sigma=3.0))
    return s


@pytest.mark.parametrize("spec,armed", [
    ([(2, 3, "fp32", False), (3, 3, "tf32", True), (2, 2, "bf16", False)], 1),
    ([(2, 3, "fp64", False), (3, 3, "tf32", True), (2, 2, "bf16", False)], 2),
    # a member above half of the L2: two clusters, the small members first
    ([(3, 22, "fp32", True), (2, 3, "tf32", False)], 1)])
def test_member_time_out_is_reported(spec, armed):
    from paper_2006_02551_gb300 import Group, WadgError
    from paper_2006_02551_gb300.wadg import WADG_ETIMEOUT
    members = [member(*m) for m in spec]
    rng = np.random.default_rng(1)
    q0 = [rng.normal(size=s.state_shape()) for s in members]
    dts = [s.stable_dt(0.5) for s in members]
    g = Group(members)

    def run():
        for s, q in zip(members, q0):
            s.set_state(q, 0.0)
        g.run_steps(3, dts)
        return [s.get_state()[0] for s in members]

    clean = run()
    members[armed].arm_wait_timeout()
    with pytest.raises(WadgError) as err:
        run()
    assert err.value.status == WADG_ETIMEOUT
    assert f"member {armed}" in str(err.value)
    for a, b in zip(run(), clean):
        assert np.array_equal(a, b)
    members[armed].set_state(q0[armed], 0.0)
    members[armed].run_steps(1, dts[armed])   # no flag of the group's call is left
    g.close()
    for s in members:
        s.close()
