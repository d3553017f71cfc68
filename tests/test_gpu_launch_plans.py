"""What a launch plan says is what runs: a mixed block count that happens to be the band's tile count is a
block count, the band's own entry selects the band and nothing else, and a closed box takes the built-in
shapes whatever is set."""
import numpy as np
import pytest

from paper_2211_10698_gb300 import ccm, inputs as I

pytestmark = pytest.mark.gpu


def _case(nx, ny, precision, degree=3, autotune=0, bc=None):
    c = I.make_case("plan", nx, ny, (-2.0, 6.0, -2.0, 2.0), I.Geometry(kind=I.GEOM_CIRCLE, cx=0.1, cy=-0.05, r=0.5), re=100.0,
                    cfl=0.5, lref=1.0, bc=bc)
    c.precision, c.autotune, c.tol_p = precision, autotune, 1e-10
    c.precond, c.cheb_degree = ("chebyshev", degree) if precision == "mixed" and degree > 1 else ("jacobi", 1)
    return c


def _phi(g, rhs):
    g.set_field(ccm.CCM_F_PHI, np.zeros(g.shape))
    assert g.solve_pressure(rhs)["converged"]
    return g.get_field(ccm.CCM_F_PHI)


@pytest.mark.parametrize("nx,ny", [(256, 128), (1024, 256)])
def test_block_counts_and_the_band(nx, ny):
    # whatever tuning chose here, the band's tile count is the one number above CCM_PLAN_BAND that is taken
    g = ccm.Case(_case(nx, ny, "mixed"))
    rhs = np.random.default_rng(0).standard_normal(g.shape)
    built_in = _phi(g, rhs)  # the band
    band = []
    for n in range(1, 305):
        try:
            g.set_launch_plan((0, 0, 0, 0, ccm.CCM_PLAN_BAND + n, 0, 0))
            band.append(n)
        except ccm.CcmError as e:
            assert e.status == ccm.CCM_E_INVALID
    assert len(band) == 1, band
    g.set_launch_plan((0, 0, 0, 0, ccm.CCM_PLAN_BAND + band[0], 0, 0))
    assert g.launch_plan() == (0, 0, 0, 0, ccm.CCM_PLAN_BAND + band[0], 0, 0)
    assert np.array_equal(_phi(g, rhs), built_in)
    for blocks in (band[0], band[0] + 1):
        g.set_launch_plan((0, 0, 0, 0, blocks, 0, 0))
        assert g.launch_plan() == (0, 0, 0, 0, blocks, 0, 0)
        assert not np.array_equal(_phi(g, rhs), built_in)  # other sums: the kernel with a barrier per step
    g.close()


@pytest.mark.parametrize("nx,ny,degree,fits", [(2048, 1024, 1, True), (2048, 1024, 3, True), (2048, 1024, 4, False),
                                               (1792, 952, 8, True), (2048, 1024, 8, False), (2304, 1152, 1, False)])
def test_where_the_band_ends(nx, ny, degree, fits):
    """Region rows are at most 15 warps of 9: tile rows and twice the degree."""
    g = ccm.Case(_case(nx, ny, "mixed", degree))
    taken = 0
    for n in range(1, 305):
        try:
            g.set_launch_plan((0, 0, 0, 0, ccm.CCM_PLAN_BAND + n, 0, 0))
            taken += 1
        except ccm.CcmError:
            pass
    g.close()
    assert taken == (1 if fits else 0)


def test_the_band_is_no_fp64_or_closed_box_plan():
    for c in (_case(256, 128, "fp64"), _case(256, 128, "mixed", bc=I.closed_box_bc())):
        g = ccm.Case(c)
        for n in range(1, 305):
            with pytest.raises(ccm.CcmError):
                g.set_launch_plan((0, 0, 0, 0, ccm.CCM_PLAN_BAND + n, 0, 0))
        g.close()


@pytest.mark.parametrize("plan", [(32, 8, 8, 128, 0, 0, 1), (64, 16, 4, 32, 0, 0, 0), (0, 0, 0, 0, 0, 8, 0)])
def test_a_closed_box_takes_the_built_in_shapes(plan):
    g = ccm.Case(_case(256, 128, "fp64", bc=I.closed_box_bc()))
    rhs = np.random.default_rng(0).standard_normal(g.shape)
    built_in = _phi(g, rhs)
    g.set_launch_plan(plan)
    assert np.array_equal(_phi(g, rhs), built_in)
    g.close()
