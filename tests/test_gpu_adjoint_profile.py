"""The FP32 profile derivatives against the FP64 context's where an error that
every element repeats shows: 16,464 elements, N = 4, the compact rule, smooth
waves.  The sums over the mesh average independent roundings out, but not the
FP32 rounding of the volume rule's coefficients, which all elements share.
Bound on the median over 24 meshes and excitations of the relative error of
dJ/dsigma_max: ten roundings (2^-24 each)."""
import numpy as np
import pytest

from synthetic import PmlProfile, compact_rule, cube_tet_mesh

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2006_02551_gb300 import build
    build.build()


def waves(N, v, e, rng):
    """Three plane waves of random direction and phase in E and H."""
    lat = np.array([(N - i - j - k, i, j, k) for k in range(N + 1) for j in range(N + 1 - k)
                    for i in range(N + 1 - k - j)]) / N
    x = np.einsum("na,kad->knd", lat, v[e])
    q = np.zeros((1, e.shape[0], 12, lat.shape[0]))
    for _ in range(3):
        k = rng.normal(size=3)
        k /= np.linalg.norm(k)
        p = np.cross(k, rng.normal(size=3))
        p /= np.linalg.norm(p)
        s = np.sin(x @ (k * rng.uniform(2.0, 6.0)) + rng.uniform(0.0, 6.28))
        q[0, :, :3] += p[None, :, None] * s[:, None]
        q[0, :, 3:6] += np.cross(k, p)[None, :, None] * s[:, None]
    return q


def test_repeated_rounding_of_the_rule():
    from paper_2006_02551_gb300 import Solver
    N = 4
    prof = PmlProfile(u0=0.8, L=0.2, sigma_max=40.0, p_sigma=3.0)
    errs = []
    for seed in range(24):
        rng = np.random.default_rng(100 + seed)
        v, e = cube_tet_mesh(14, 0.2, seed)
        eps = rng.uniform(1.0, 4.0, e.shape[0])
        probes = rng.uniform(-0.6, 0.6, (8, 3))
        q0 = waves(N, v, e, rng)
        grad = {}
        for prec in ("fp64", "fp32"):
            s = Solver(N, prec)
            s.set_quadrature(compact_rule(N))
            s.set_mesh(v, e)
            s.set_materials(eps)
            s.set_pml(prof)
            s.set_probes(probes)
            s.set_state(q0, 0.0)
            grad[prec] = s.adjoint(12, s.stable_dt(1.0), 12)[2][0]
            s.close()
        errs.append(np.linalg.norm(grad["fp32"] - grad["fp64"]) / np.linalg.norm(grad["fp64"]))
    print("relative errors of dJ/dsigma_max:", ["%.1e" % x for x in sorted(errs)])
    assert np.median(errs) < 10 * 2.0 ** -24, errs
