"""Closed boxes near rounding: the one-barrier kernels solve the singular system without projecting every
residual, and have to converge as the general kernel does, which projects each (the Chebyshev setting of
degree 1 is Jacobi on that kernel): to tolerances of a few units of rounding, and with a right-hand side
whose mean, which is taken off first, is a million times its variation (where the general kernel, which
counts what rounding leaves of the mean in its residual, does not: the variation alone is its measure)."""
import ctypes

import numpy as np
import pytest

from paper_2211_10698_gb300 import ccm, inputs as I

pytestmark = pytest.mark.gpu


def _case(nx, ny, body, tol, general=False):
    geom = I.Geometry(kind=I.GEOM_CIRCLE, cx=0.5, cy=0.5 * ny / nx, r=0.11) if body else I.Geometry()
    c = I.make_case("closed", nx, ny, (0.0, 1.0, 0.0, ny / nx), geom, re=100.0, cfl=0.5, lref=1.0, bc=I.closed_box_bc(lid=1.0))
    c.autotune, c.tol_p, c.max_iter_p = 0, tol, 20000
    c.precond, c.cheb_degree = ("chebyshev", 1) if general else ("jacobi", 1)
    return c


def _rhs(c, kind):
    x, y = np.linspace(0.0, 1.0, c.shape[1]), np.linspace(0.0, 1.0, c.shape[0])[:, None]
    s = np.exp(-((x - 0.3) / 0.1) ** 2 - ((y - 0.6) / 0.2) ** 2) - 0.7 * np.exp(-((x - 0.8) / 0.2) ** 2 - ((y - 0.2) / 0.1) ** 2)
    return 1.0 + 1e-6 * s if kind == "large mean" else s


def _residual(o, rhs, phi):
    b = np.where(o.active, rhs - rhs[o.active].mean(), 0.0)
    return np.linalg.norm((b - o.poisson(phi))[o.active]) / np.linalg.norm(b)


CASES = [(64, 64, False, "smooth", 1e-14), (150, 33, False, "smooth", 1e-14), (192, 192, False, "smooth", 1e-13),
         (192, 192, True, "smooth", 1e-13), (64, 64, False, "large mean", 1e-10), (192, 192, False, "large mean", 1e-10),
         (192, 192, True, "large mean", 1e-10), (1100, 1100, False, "smooth", 1e-11)]


@pytest.mark.parametrize("nx,ny,body,kind,tol", CASES)
def test_closed_box_converges_like_the_projected_iteration(orc, nx, ny, body, kind, tol):
    got = []
    for general in (False, True):
        # the residual of CG goes down in waves, and which of them first meets a tolerance is a matter of the
        # last bit of a dip: the general kernel is given half the tolerance
        c = _case(nx, ny, body, 0.5 * tol if general else tol, general)
        g = ccm.Case(c)
        rhs = _rhs(c, "smooth" if general else kind)
        st = g.solve_pressure(rhs)
        assert st["converged"], (general, st)
        phi = g.get_field(ccm.CCM_F_PHI)
        o = orc.Oracle(c)
        got.append((st["iters"], _residual(o, rhs, phi)))
        # zero mean to the rounding of the sum
        assert abs(phi[o.active].sum()) <= 1e-11 * np.abs(phi[o.active]).sum()
        g.close()
    (it, res), (it0, res0) = got
    assert it <= 1.03 * it0 + 3, got
    # the mean is taken off to a unit or two of rounding of its value in every cell, 4.4e-16, and the
    # variation's root mean square is above 2e-7
    assert res <= 2.0 * res0 + tol + (2.2e-9 if kind == "large mean" else 0.0), got


@pytest.mark.parametrize("nx,ny,kind,tol", [(192, 192, "smooth", 1e-13), (64, 64, "large mean", 1e-10)])
def test_allocation_free_solve(nx, ny, kind, tol):
    import torch

    g0 = ccm.Case(_case(nx, ny, False, 0.5 * tol, True))
    c = _case(nx, ny, False, tol)
    rhs = _rhs(c, kind)
    it0 = g0.solve_pressure(_rhs(c, "smooth"))["iters"]
    g = ccm.Case(c)
    _, pitch = g.device_ptr(ccm.CCM_F_PHI)
    b = torch.zeros((c.shape[0], pitch), dtype=torch.float64, device="cuda")
    b[:, :c.shape[1]] = torch.from_numpy(rhs).cuda()
    phi = torch.zeros_like(b)
    torch.cuda.synchronize()
    st = ccm.ccm_solve_stats()
    assert ccm.lib().ccm_solve_pressure_noalloc(g.h, ctypes.c_void_p(b.data_ptr()), ctypes.c_void_p(phi.data_ptr()),
                                                ctypes.byref(st)) == ccm.CCM_OK
    assert st.iters <= 1.03 * it0 + 3, (st.iters, it0)
    g0.close()
    g.close()
