"""A uniform and a stretched mesh of one size, tuned in one process in either order: neither takes over the
other's launch shape.  At these sizes the mixed band tiles fit the uniform mesh only (a stretched one keeps
coefficients of every row in shared memory)."""
import numpy as np
import pytest

from paper_2211_10698_gb300 import ccm, inputs as I

pytestmark = pytest.mark.gpu


def _case(nx, ny, stretched):
    box, kw = (-2.0, 6.0, -2.0, 2.0), {}
    if stretched:
        for key, n, lo, hi in (("xf", nx, *box[:2]), ("yf", ny, *box[2:])):
            f = np.concatenate([[0.0], np.cumsum(1.0 + 0.5 * np.sin(np.arange(n) / n * 3.0))])
            f = lo + f * ((hi - lo) / f[-1])
            f[0], f[-1] = lo, hi
            kw[key] = f
    c = I.make_case("tune", nx, ny, box, I.Geometry(kind=I.GEOM_CIRCLE, cx=0.1, cy=-0.05, r=0.5), re=100.0, cfl=0.5, lref=1.0, **kw)
    c.precision, c.precond, c.cheb_degree, c.autotune = "mixed", "chebyshev", 3, 1
    return c


@pytest.mark.parametrize("nx,ny,order", [(1500, 1100, (False, True)), (1496, 1104, (True, False))])
def test_tuned_shapes(nx, ny, order):
    plans = {}
    for stretched in order:
        g = ccm.Case(_case(nx, ny, stretched))
        plans[stretched] = g.launch_plan()
        g.close()
    assert plans[False] != plans[True], plans
    for stretched in order:  # each finds its own again
        g = ccm.Case(_case(nx, ny, stretched))
        assert g.launch_plan() == plans[stretched]
        g.close()
