"""wadg_memory_report against the bytes that a context holds
(wadg_set_memory_limit): the operators column is every operator and orbit
table, the state, samples and geometry columns every per-element buffer but the
vertices (96 bytes) and the element order (4 bytes)."""
import pytest

from synthetic import PmlProfile, compact_rule, cube_tet_mesh

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2006_02551_gb300 import build
    build.build()


@pytest.mark.parametrize("prec,compact,kappa", [
    ("fp64", False, 1.0), ("fp64", True, 2.0), ("fp32", False, 2.0), ("fp32", True, 1.0),
    ("tf32", True, 1.0), ("bf16", False, 1.0)])
def test_report_covers_what_is_held(prec, compact, kappa):
    from paper_2006_02551_gb300 import Solver
    s = Solver(3, prec, n_batch=2)
    if compact:
        s.set_quadrature(compact_rule(3))
    held0 = s.set_memory_limit(0)
    counters = 8 + 8 + 4 + 8 + 8 * 2   # time, step, two flag words, objective
    assert s.memory_report()["operators"] == held0 - counters
    v, e = cube_tet_mesh(3, 0.1, 1)
    s.set_mesh(v, e)
    s.set_pml(PmlProfile(u0=0.5, L=0.5, sigma_max=20.0, p_sigma=3.0, kappa_max=kappa))
    r = s.memory_report()
    assert (r["state"] + r["pml_coeff"] + r["geometry"] + 100 * e.shape[0]
            == s.set_memory_limit(0) - held0)
    s.close()
