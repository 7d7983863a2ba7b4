"""Time-outs of the CUDA-core kernels' bounded waits, in the diagnostic build
(-DWADG_CHECKED), where a request can be armed on FP64 and FP32 contexts: one
block waits for bytes that no copy brings, its wait gives up after about a
second, the call returns WADG_ETIMEOUT, and the context steps bit for bit as
before afterwards.  Cases: the launch of both classes with its chained stages
(small meshes), one launch per class (beyond one wave of blocks, and the
single-stage and allocation-free calls), several tiles per block, both rules,
kappa, grouped variant kernels and per-item launches, and the FP32 reverse
stage.  Nothing here faults, traps or waits without a limit."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r'''
import time
import numpy as np
from paper_2006_02551_gb300 import Group, Solver, WadgError, wadg
assert wadg.LIB_PATH.endswith("libwadg_checked.so"), wadg.LIB_PATH
from synthetic import Dipole, PmlProfile, compact_rule, cube_tet_mesh


def solver(prec, N, n, compact, kappa=1.0):
    v, e = cube_tet_mesh(n, 0.15, 3)
    s = Solver(N, prec)
    if compact:
        s.set_quadrature(compact_rule(N))
    s.set_mesh(v, e)
    s.set_pml(PmlProfile(u0=0.5, L=0.5, sigma_max=10.0, p_sigma=2.0, kappa_max=kappa))
    s.set_probes([(0.1, 0.2, 0.3)])
    q0 = np.random.default_rng(n).normal(size=s.state_shape())
    q0[:, :, 6:] = 0.0
    return s, q0


def timed_out(call):
    t0 = time.perf_counter()
    try:
        call()
    except WadgError as err:
        assert err.status == wadg.WADG_ETIMEOUT, err
        assert time.perf_counter() - t0 < 20.0
        return True
    return False


for prec, N, n, compact, kappa in (("fp64", 3, 3, True, 1.0), ("fp64", 4, 8, False, 1.0),
                                   ("fp32", 2, 4, False, 1.0), ("fp32", 3, 20, True, 2.0),
                                   ("fp32", 5, 4, False, 1.0)):
    s, q0 = solver(prec, N, n, compact, kappa)
    dt = s.stable_dt(0.5)
    calls = [lambda: s.run_steps(2, dt), lambda: s.run_steps_noalloc(2, dt),
             lambda: [s.rk_stage(i, 0.0, dt) for i in range(5)]]
    for call in calls:
        s.set_state(q0, 0.0)
        call()
        clean = s.get_state()[0]
        s.set_state(q0, 0.0)
        s.arm_wait_timeout()
        assert timed_out(call), (prec, N, n)
        s.set_state(q0, 0.0)
        call()
        assert np.array_equal(s.get_state()[0], clean), (prec, N, n)
    s.close()
    print("stepping", prec, N, n, flush=True)

for per_item in (False, True):
    pairs = [solver("fp32", N, n, False) for N, n in ((2, 8), (3, 6), (2, 5))]
    members = [p[0] for p in pairs]
    dts = [m.stable_dt(0.5) for m in members]
    g = Group(members)
    g.set_tuning(per_item=per_item)
    def run():
        for m, q in pairs:
            m.set_state(q, 0.0)
        g.run_steps(2, dts)
        return [m.get_state()[0] for m in members]
    clean = run()
    members[2].arm_wait_timeout()
    assert timed_out(run), per_item
    assert all(np.array_equal(a, b) for a, b in zip(run(), clean)), per_item
    g.close()
    for m in members:
        m.close()
    print("group", per_item, flush=True)

for N, n, compact in ((2, 3, True), (3, 6, False)):
    s, q0 = solver("fp32", N, n, compact)
    dt = s.stable_dt(0.5)
    s.set_state(q0, 0.0)
    clean = s.adjoint(3, dt, 2)
    s.set_state(q0, 0.0)
    s.arm_wait_timeout()
    s.arm_wait_timeout()                     # the reverse stage
    assert timed_out(lambda: s.adjoint(3, dt, 2)), N
    s.set_state(q0, 0.0)
    again = s.adjoint(3, dt, 2)
    for a, b in zip(again, clean):           # (shared-memory sums in any order)
        assert np.allclose(a, b, rtol=1e-5, atol=1e-6 * np.abs(b).max()), N
    s.close()
    print("adjoint", N, n, flush=True)
print("waits ok")
'''


def test_cuda_core_waits_time_out():
    from paper_2006_02551_gb300 import build
    lib = build.build(checked=True)
    env = dict(os.environ, WADG_LIB=lib)
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, env=env, capture_output=True,
                       text=True, timeout=600)
    assert r.returncode == 0 and "waits ok" in r.stdout, r.stdout + r.stderr
