"""A zero right-hand side has the solution zero, whatever warm start the solve is given: every kernel
that serves a pressure solve, alone and batched, in open and closed boxes.  The oracle says the same."""
import ctypes

import numpy as np
import pytest

from paper_2211_10698_gb300 import ccm, inputs as I

pytestmark = pytest.mark.gpu

OPEN = ((I.BC_DIRICHLET, I.BC_OUTFLOW, I.BC_OUTFLOW, I.BC_OUTFLOW), (0.0,) * 4, (0.0,) * 4)


def _case(box, precision="fp64", degree=1, nx=128, ny=64):
    bc = OPEN if box == "open" else I.closed_box_bc()
    c = I.make_case("still", nx, ny, (-2.0, 6.0, -2.0, 2.0), I.Geometry(kind=I.GEOM_CIRCLE, cx=0.1, cy=-0.05, r=0.5), re=100.0,
                    cfl=0.5, lref=1.0, bc=bc)
    c.precision, c.autotune = precision, 0
    c.precond, c.cheb_degree = ("chebyshev", degree) if degree > 1 else ("jacobi", 1)
    return c


def _warm(c, seed=0):
    w = np.zeros(c.shape)
    w[1:-2, 1:-2] = np.random.default_rng(seed).standard_normal((c.ny, c.nx))
    return w


# (box, precision, Chebyshev degree, launch plan)
SOLVES = [("open", "fp64", 1, None),                            # resident tiles
          ("open", "fp64", 1, (32, 8, 4, 32, 0, 0, 0)),         # tiles in global memory
          ("open", "fp64", 1, (0, 0, 0, 0, 0, 8, 0)),           # one cluster
          ("open", "fp64", 3, None),                            # general kernel
          ("closed", "fp64", 1, None),
          ("closed", "fp64", 3, None),
          ("open", "mixed", 1, None), ("open", "mixed", 3, None),  # band tiles
          ("open", "mixed", 1, (0, 0, 0, 0, 64, 0, 0)),         # a barrier per phase
          ("open", "mixed", 3, (64, 16, 2, 8, 0, 0, 0)),        # one-barrier tiles
          ("open", "mixed", 3, (64, 16, 2, 8, 0, 0, 1)),
          ("closed", "mixed", 1, None)]                         # refinement from the host


@pytest.mark.parametrize("box,precision,degree,plan", SOLVES)
def test_solve(orc, box, precision, degree, plan):
    c = _case(box, precision, degree)
    g = ccm.Case(c)
    if plan:
        g.set_launch_plan(plan)
    g.set_field(ccm.CCM_F_PHI, _warm(c))
    st = g.solve_pressure(np.zeros(c.shape))
    assert st["converged"] and st["rel_res"] == 0.0, st
    assert not g.get_field(ccm.CCM_F_PHI).any()
    assert not orc.Oracle(c).solve_poisson(np.zeros(c.shape), _warm(c))[0].any()
    # and the next right-hand side is solved as ever
    rhs = _warm(c, 1)
    assert g.solve_pressure(rhs)["converged"]
    g.close()


@pytest.mark.parametrize("box,degree", [("open", 1), ("open", 3), ("closed", 1)])
def test_noalloc(box, degree):
    import torch

    c = _case(box, "fp64", degree)
    g = ccm.Case(c)
    rows, cols = g.shape
    _, pitch = g.device_ptr(ccm.CCM_F_PHI)
    rhs = torch.zeros((rows, pitch), dtype=torch.float64, device="cuda")
    phi = torch.zeros_like(rhs)
    phi[:, :cols] = torch.from_numpy(_warm(c)).cuda()
    torch.cuda.synchronize()
    st = ccm.ccm_solve_stats()
    assert ccm.lib().ccm_solve_pressure_noalloc(g.h, ctypes.c_void_p(rhs.data_ptr()), ctypes.c_void_p(phi.data_ptr()),
                                                ctypes.byref(st)) == ccm.CCM_OK
    assert not phi[1:-2, 1:cols - 2].any()
    g.close()


# (boxes, precision, degree, sizes): resident tiles, vectors in global memory, the general batch, the
# mixed batch, the refinement from the host
BATCHES = [("open", "fp64", 1, [(128, 64), (61, 37)]), ("open", "fp64", 1, [(1024, 512), (1024, 300)]),
           ("closed", "fp64", 1, [(128, 64), (61, 37)]), ("open", "mixed", 1, [(128, 64), (61, 37)]),
           ("open", "mixed", 4, [(128, 64), (61, 37)]), ("closed", "mixed", 1, [(128, 64), (61, 37)])]


@pytest.mark.parametrize("box,precision,degree,sizes", BATCHES)
def test_fluid_at_rest_stays_at_rest(box, precision, degree, sizes):
    """Steps of a fluid at rest with the Phi of an earlier flow: alone and in a batch."""
    def still(nx, ny):
        c = ccm.Case(_case(box, precision, degree, nx, ny))
        for f in (ccm.CCM_F_U, ccm.CCM_F_V, ccm.CCM_F_P):
            c.set_field(f, np.zeros(c.shape))
        c.set_field(ccm.CCM_F_PHI, _warm(c.spec))
        return c

    cases = [still(*s) for s in sizes]
    b = ccm.Batch(len(cases))
    for c in cases:
        b.add(c)
    assert all(s["converged"] for s in b.step(1))
    b.close()
    alone = still(*sizes[0])
    assert alone.step(1)["converged"]
    for c in cases + [alone]:
        for f in (ccm.CCM_F_U, ccm.CCM_F_V, ccm.CCM_F_P):
            assert not c.get_field(f).any(), (c.spec.nx, f)
        c.close()
