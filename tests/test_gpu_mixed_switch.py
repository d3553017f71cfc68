"""The mixed kernels share a case's work arrays and lay them out differently (the band tiles' quads lie one
element off the others').  Whatever ran before, a solve gives the bits of a fresh case's."""
import numpy as np
import pytest

from paper_2211_10698_gb300 import ccm, inputs as I

pytestmark = pytest.mark.gpu

PLANS = {"band": (0,) * 7, "barrier per step": (0, 0, 0, 0, 64, 0, 0), "tiles": (32, 8, 8, 104, 0, 0, 0),
         "resident tiles": (32, 8, 8, 104, 0, 0, 1)}


def _case(degree):
    c = I.make_case("switch", 243, 101, (-2.0, 6.0, -2.0, 2.0), I.Geometry(kind=I.GEOM_CIRCLE, cx=0.1, cy=-0.05, r=0.5), re=100.0,
                    cfl=0.5, lref=1.0)
    c.precision, c.autotune, c.tol_p = "mixed", 0, 1e-10
    c.precond, c.cheb_degree = ("chebyshev", degree) if degree > 1 else ("jacobi", 1)
    return c


def _solve(g, plan, rhs):
    g.set_launch_plan(plan)
    g.set_field(ccm.CCM_F_PHI, np.zeros(g.shape))
    assert g.solve_pressure(rhs)["converged"]
    return g.get_field(ccm.CCM_F_PHI)


@pytest.mark.parametrize("degree", [1, 3])
def test_any_kernel_after_any_other(degree):
    c = _case(degree)
    rhs = np.random.default_rng(degree).standard_normal(c.shape)
    fresh = {}
    for name, plan in PLANS.items():
        g = ccm.Case(c)
        fresh[name] = _solve(g, plan, rhs)
        g.close()
    g = ccm.Case(c)
    for first in PLANS:
        for then in PLANS:
            _solve(g, PLANS[first], rhs[::-1].copy())
            assert np.array_equal(_solve(g, PLANS[then], rhs), fresh[then]), (first, then)
    g.close()


@pytest.mark.parametrize("degree", [1, 4])
def test_a_batch_after_band_solves(degree):
    def step(used):
        g = ccm.Case(_case(degree))
        if used:
            _solve(g, PLANS["band"], np.random.default_rng(1).standard_normal(g.shape))
            g.set_field(ccm.CCM_F_PHI, np.zeros(g.shape))
        b = ccm.Batch(1)
        b.add(g)
        b.step(2)
        out = [g.get_field(f) for f in (ccm.CCM_F_U, ccm.CCM_F_V, ccm.CCM_F_P)]
        b.close()
        g.close()
        return out

    for a, b in zip(step(False), step(True)):
        assert np.array_equal(a, b)
