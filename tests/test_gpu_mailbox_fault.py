"""One block of a resident solve sends its neighbours nothing: their waits run out while the other blocks
still iterate.  Every block leaves the launch, the step returns CCM_E_TIMEOUT, and the case steps on as
before once the fault is cleared and a checkpoint restored."""
import ctypes
import time

import numpy as np
import pytest

from paper_2211_10698_gb300 import ccm, inputs as I

pytestmark = pytest.mark.gpu

STATE = (ccm.CCM_F_U, ccm.CCM_F_V, ccm.CCM_F_P, ccm.CCM_F_PHI, ccm.CCM_F_CONV_U, ccm.CCM_F_CONV_V, ccm.CCM_F_STEP)


# the silent block at a corner and inside; FP64 tiles of 128, 256 and 512 threads; one and several rows
# per warp of the band tiles
@pytest.mark.parametrize("silent", [0, 7, 17])
@pytest.mark.parametrize("precision,degree,nx,ny", [("fp64", 1, 128, 64), ("fp64", 1, 256, 128), ("fp64", 1, 1024, 512),
                                                    ("mixed", 1, 256, 128), ("mixed", 3, 256, 128), ("mixed", 3, 1024, 512)])
def test_silent_block(precision, degree, nx, ny, silent):
    case = I.small_cylinder(nx=nx, ny=ny, box=(-2.0, 6.0, -2.0, 2.0), r=0.5, cx=0.0, cy=0.0)
    case.precision, case.precond, case.cheb_degree = precision, "chebyshev" if degree > 1 else "jacobi", degree
    case.autotune = 0
    g = ccm.Case(case)
    g.step(1)
    ck = {f: g.get_field(f).copy() for f in STATE}
    L, st = ccm.lib(), ccm.ccm_step_stats()
    assert L.ccm_set_barrier_fault(g.h, 1_000_000, -1) == ccm.CCM_OK  # about 0.5 ms per wait
    assert L.ccm_set_mailbox_fault(g.h, silent) == ccm.CCM_OK
    t0 = time.time()
    status = L.ccm_step(g.h, 1, ctypes.byref(st))
    assert status == ccm.CCM_E_TIMEOUT, (ccm.STATUS_NAMES[status], L.ccm_last_error())
    assert time.time() - t0 < 10.0
    assert L.ccm_set_barrier_fault(g.h, 0, -1) == ccm.CCM_OK and L.ccm_set_mailbox_fault(g.h, -1) == ccm.CCM_OK
    for f in STATE:
        g.set_field(f, ck[f])
    assert g.step(1)["converged"]
    ref = ccm.Case(case)
    ref.step(2)
    for f in (ccm.CCM_F_U, ccm.CCM_F_V, ccm.CCM_F_P, ccm.CCM_F_PHI):
        assert np.array_equal(g.get_field(f), ref.get_field(f)), f
    assert L.ccm_set_mailbox_fault(g.h, -2) == ccm.CCM_E_INVALID
    g.close()
    ref.close()
