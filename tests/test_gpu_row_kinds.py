"""Rows whose face coefficients differ from the uniform grid's by the rounding of the abscissas only
take the constant stencil: grids whose spacing is no dyadic fraction, boxes away from the origin, one
row of cells many spacings from it.  The residual of each solution under the oracle's operator, which
has the rounded coefficients, meets the tolerance of the solve."""
import numpy as np
import pytest

from paper_2211_10698_gb300 import ccm, inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed", "mixed, a barrier per step"])
@pytest.mark.parametrize("nx,ny,x0", [(61, 37, 0.0), (250, 121, 0.0), (333, 97, 30.0), (701, 333, 0.0)])
def test_uncut_rows_of_rounded_grids(orc, nx, ny, x0, precision):
    box = (x0 - 2.0, x0 + 6.0, -2.0, 2.0)
    c = I.make_case("rounded", nx, ny, box, I.Geometry(kind=I.GEOM_CIRCLE, cx=x0 + 0.1, cy=-0.05, r=0.5), re=100.0, cfl=0.5, lref=1.0)
    c.precision, c.tol_p, c.autotune = precision.split(",")[0], 1e-10, 0
    o = orc.Oracle(c)
    rhs = np.random.default_rng(nx).standard_normal(c.shape) * o.active
    g = ccm.Case(c)
    if precision != c.precision:
        g.set_launch_plan((0, 0, 0, 0, 304, 0, 0))
    st = g.solve_pressure(rhs)
    assert st["converged"], st
    res = rhs - o.poisson(g.get_field(ccm.CCM_F_PHI))
    assert np.linalg.norm(res[o.active]) <= 1.05 * c.tol_p * np.linalg.norm(rhs)
    g.close()
