"""Uniform FP64 grids whose abscissas are rounded (a spacing that is no dyadic fraction, a box away from the
origin): solution, projection and capacities share one operator, so a solve meets its tolerance under the
case's own operator wherever the box lies, and a step leaves the same divergence.

The residual of a solve whose recurrence has met the tolerance is the recurrence's, plus the rounding of
x and K x, which does not depend on the box's place: the box at the origin sets the scale."""
import numpy as np
import pytest

from paper_2211_10698_gb300 import ccm, inputs as I

pytestmark = pytest.mark.gpu


def _open(nx, ny, x0):
    return I.make_case("far", nx, ny, (x0 - 2.0, x0 + 6.0, -2.0, 2.0), I.Geometry(kind=I.GEOM_CIRCLE, cx=x0 + 0.1, cy=-0.05, r=0.5),
                       re=100.0, cfl=0.5, lref=1.0)


def _closed(nx, ny, x0):
    return I.make_case("far", nx, ny, (x0, x0 + 1.0, 0.0, ny / nx), I.Geometry(), re=100.0, cfl=0.5, lref=1.0,
                       bc=I.closed_box_bc(lid=1.0))


def _smooth(c):
    x, y = np.linspace(0.0, 1.0, c.shape[1]), np.linspace(0.0, 1.0, c.shape[0])[:, None]
    return np.exp(-((x - 0.3) / 0.1) ** 2 - ((y - 0.6) / 0.2) ** 2) - 0.7 * np.exp(-((x - 0.8) / 0.2) ** 2 - ((y - 0.2) / 0.1) ** 2)


def _residual(make, nx, ny, x0):
    c = make(nx, ny, x0)
    c.tol_p, c.autotune = 1e-11, 0
    g = ccm.Case(c)
    b = _smooth(c)
    assert g.solve_pressure(b)["converged"]
    one = np.zeros(c.shape)
    one[1:-2, 1:-2] = 1.0
    act = (g.apply(ccm.CCM_OP_POISSON_DIAG, nout=1) != 0) & (one != 0)
    act &= g.cap("p", "V") > 0
    if make is _closed:
        b = b - b[act].mean()
    r = (b - g.apply(ccm.CCM_OP_POISSON, g.get_field(ccm.CCM_F_PHI), nout=1))[act]
    g.close()
    return np.linalg.norm(r) / np.linalg.norm(b[act])


@pytest.mark.parametrize("make,nx,ny", [(_open, 701, 333), (_open, 250, 121), (_closed, 200, 200)])
def test_residual_under_the_cases_own_operator(make, nx, ny):
    at = {x0: _residual(make, nx, ny, x0) for x0 in (0.0, 100.0, -1000.0)}
    assert max(at.values()) <= 2.0 * at[0.0] + 1e-11, at
    assert at[0.0] <= 1e-9, at


@pytest.mark.parametrize("x0", [0.0, 100.0, 1000.0])
def test_uncut_lengths_and_areas_are_the_grids(x0):
    c = _open(333, 97, x0)
    c.autotune = 0
    g = ccm.Case(c)
    hx, hy = 8.0 / 333, 4.0 / 97
    for grid in ("p", "u", "v"):
        v, ax, ay = (g.cap(grid, n)[1:-2, 1:-2] for n in ("V", "AX", "AY"))
        for a, h in ((v, (c.x1 - c.x0) / 333 * ((c.y1 - c.y0) / 97)), (ax, (c.y1 - c.y0) / 97), (ay, (c.x1 - c.x0) / 333)):
            near = np.abs(a - h) <= 1e-9 * h
            assert near.mean() > 0.9 and np.array_equal(a[near], np.full(near.sum(), h)), (grid, np.abs(a[near] - h).max() / h)
    assert abs(hx * hy * 333 * 97 - np.pi * 0.25 - g.cap("p", "V")[1:-2, 1:-2].sum()) < 1e-2
    g.close()


@pytest.mark.parametrize("x0", [0.0, 100.0])
def test_a_step_leaves_the_same_divergence(x0):
    c = _open(500, 250, x0)
    c.tol_p, c.autotune = 1e-11, 0
    g = ccm.Case(c)
    st = g.step(3)
    assert st["converged"] and st["max_div"] <= 1e-9, st
    g.close()


def test_mixed_cases_keep_their_lengths(orc):
    c = _open(333, 97, 30.0)
    c.precision, c.autotune = "mixed", 0
    g, o = ccm.Case(c), orc.Oracle(c)
    a, b = g.cap("p", "AX")[1:-2, 1:-2], o.cap("p", "AX")[1:-2, 1:-2]
    assert np.abs(a - b).max() <= 1e-14 * np.abs(b).max()
    g.close()
