"""Device memory of a case (ccm_case_bytes, on the CPU): the mailboxes of the FP64 tiles are carved for the
cases that can use them only."""
import pytest

from paper_2211_10698_gb300 import ccm, inputs as I


def _bytes(nx, ny, precision, bc=None):
    c = I.make_case("bytes", nx, ny, (0.0, 2.0, 0.0, 1.0), I.Geometry(), re=100.0, cfl=0.5, lref=1.0, bc=bc)
    return ccm.case_bytes(c, precision=precision)


@pytest.mark.parametrize("nx,ny", [(48, 24), (129, 63), (1026, 513)])
def test_mailboxes(nx, ny):
    mixed, fp64 = _bytes(nx, ny, "mixed"), _bytes(nx, ny, "fp64")
    # slots of 16 bytes, two per ring cell: the rings of the smallest tiles (one row, 32 columns) at least
    tiles = min(-(-nx // 32) * ny, 480)
    assert fp64 - mixed >= 16 * 4 * tiles * 32
    assert fp64 - mixed < 0.5 * mixed
    assert _bytes(nx, ny, "mixed", I.closed_box_bc()) == mixed
    if nx % 3 == 0:
        assert _bytes(nx, ny, "fp64", I.periodic_bc(True, False)) == mixed
