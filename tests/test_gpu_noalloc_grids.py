"""Grids whose smallest tiles are wide and flat, so that the rings of the tiles outgrow the mailboxes of
the allocation-free solve's fixed scratch: the solve takes another plan and gives the case's own solution.
And tile plans whose tiles are higher than the grid, which a caller may set: the case's mailboxes hold them."""
import ctypes

import numpy as np
import pytest

from paper_2211_10698_gb300 import ccm, inputs as I

pytestmark = pytest.mark.gpu


def _case(nx, ny):
    c = I.make_case("grid", nx, ny, (0.0, nx / 8.0, 0.0, ny / 8.0), I.Geometry(), re=100.0, cfl=0.5, lref=1.0)
    c.autotune, c.tol_p = 0, 1e-9
    return c


@pytest.mark.parametrize("nx,ny", [(500, 150), (490, 136), (511, 136), (431, 152), (511, 237), (4000, 19), (3841, 19), (4096, 19)])
def test_flat_tiles(nx, ny):
    import torch

    c = _case(nx, ny)
    g = ccm.Case(c)
    rhs = np.random.default_rng(nx).standard_normal(c.shape)
    assert g.solve_pressure(rhs)["converged"]
    want = g.get_field(ccm.CCM_F_PHI)
    _, pitch = g.device_ptr(ccm.CCM_F_PHI)
    b = torch.zeros((c.shape[0], pitch), dtype=torch.float64, device="cuda")
    b[:, :c.shape[1]] = torch.from_numpy(rhs).cuda()
    phi = torch.zeros_like(b)
    torch.cuda.synchronize()
    st = ccm.ccm_solve_stats()
    status = ccm.lib().ccm_solve_pressure_noalloc(g.h, ctypes.c_void_p(b.data_ptr()), ctypes.c_void_p(phi.data_ptr()), ctypes.byref(st))
    assert status == ccm.CCM_OK, ccm.lib().ccm_last_error()
    got = phi.cpu().numpy()[:, :c.shape[1]]
    # residuals of at most 1e-9 |b| each, and K's smallest eigenvalue on these boxes is above 1e-5
    assert np.linalg.norm((got - want)[1:-2, 1:-2]) <= 2e-4 * np.linalg.norm(rhs[1:-2, 1:-2])
    g.close()


@pytest.mark.parametrize("nx,ny,tx,ty", [(13, 20, 32, 120), (4, 4, 32, 100), (40, 9, 64, 60)])
def test_tiles_higher_than_the_grid(nx, ny, tx, ty):
    c = _case(nx, ny)
    g = ccm.Case(c)
    rhs = np.random.default_rng(nx).standard_normal(c.shape)
    g.set_launch_plan((tx, ty, -(-nx // tx), -(-nx // tx), 0, 0, 1))
    assert g.solve_pressure(rhs)["converged"]
    g.close()
