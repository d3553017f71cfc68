"""The resident one-barrier FP64 solve (k_pcg_poisson_f2) at the edges of its launch rules: 128, 256
and 512 computing threads, tiles that the grid clips, tiles of one row, rings longer than a block's
threads, and meshes every row of which has coefficients of its own.  Resident and global tiles run
the same operations in the same order (a one-step rounding apart at most), and the solution meets the
tolerance under the oracle's operator."""
import numpy as np
import pytest

from paper_2211_10698_gb300 import ccm, inputs as I

pytestmark = pytest.mark.gpu


def _plan(nx, ny, tx, ty, resident):
    nbx = -(-nx // tx)
    return (tx, ty, nbx, nbx * -(-ny // ty), 0, 0, resident)


# (nx, ny, tile width, tile height): cells <= 256, <= 1024, more; clipped tiles; one row; 512 wide
SHAPES = [(128, 64, 32, 8), (70, 33, 64, 3), (70, 33, 32, 11), (260, 130, 64, 16), (260, 130, 128, 9), (530, 36, 512, 3),
          (530, 36, 256, 5), (13, 150, 32, 50)]


@pytest.mark.parametrize("stretched", [False, True])
@pytest.mark.parametrize("nx,ny,tx,ty", SHAPES)
def test_resident_tiles_at_the_edges_of_the_launch_rules(orc, nx, ny, tx, ty, stretched):
    box = (0.0, nx / 8.0, 0.0, ny / 8.0)
    geom = I.Geometry(kind=I.GEOM_CIRCLE, cx=box[1] * 0.45, cy=box[3] * 0.5, r=0.33) if min(nx, ny) >= 30 else I.Geometry()
    kw = {}
    if stretched:
        grow = lambda n: np.concatenate([[0.0], np.cumsum(1.0 + 0.5 * np.sin(np.arange(n) / n))])  # noqa: E731
        for key, n, hi in (("xf", nx, box[1]), ("yf", ny, box[3])):
            f = grow(n) * (hi / grow(n)[-1])
            f[-1] = hi
            kw[key] = f
    case = I.make_case("tiles", nx, ny, box, geom, re=50.0, cfl=0.5, lref=1.0, **kw)
    case.tol_p, case.autotune = 1e-12, 0
    o = orc.Oracle(case)
    rhs = np.random.default_rng(nx + ny).standard_normal(case.shape) * o.active
    its, phi = [], []
    for resident in (1, 0):
        g = ccm.Case(case)
        g.set_launch_plan(_plan(nx, ny, tx, ty, resident))
        st = g.solve_pressure(rhs)
        assert st["converged"], st
        its.append(st["iters"])
        phi.append(g.get_field(ccm.CCM_F_PHI))
        res = rhs - o.poisson(phi[-1])
        assert np.linalg.norm(res[o.active]) <= 1.01 * case.tol_p * np.linalg.norm(rhs)
        g.close()
    assert abs(its[0] - its[1]) <= 1
    assert np.linalg.norm(phi[0] - phi[1]) <= 1e-9 * np.linalg.norm(phi[1])


@pytest.mark.parametrize("sizes", [[(40, 24), (300, 150), (33, 61)],                 # resident tiles
                                   [(64, 32)] * 40 + [(512, 256)],                   # ... of many cases and a large one
                                   [(1024, 512), (1024, 300), (128, 64)]])           # too many cells: vectors in global memory
def test_fp64_batch_on_both_sides_of_the_resident_limit(sizes):
    """A batched FP64 step gives each case's own step (solver tolerance apart)."""
    def make(nx, ny):
        c = I.small_cylinder(nx=nx, ny=ny, box=(-2.0, 6.0, -2.0, 2.0), r=0.5, cx=0.1, cy=-0.05)
        c.tol_p, c.tol_h, c.autotune = 1e-11, 1e-12, 0
        return ccm.Case(c)

    alone, mixed = [make(*s) for s in sizes], [make(*s) for s in sizes]
    b = ccm.Batch(len(sizes))
    for c in mixed:
        b.add(c)
    for _ in range(2):
        assert all(s["converged"] for s in b.step(1))
    pairs = list(zip(alone, mixed))
    for c, m in pairs[:1] + pairs[1:][-4:]:
        c.step(2)
        for f in (ccm.CCM_F_U, ccm.CCM_F_V, ccm.CCM_F_P):
            a, got = c.get_field(f), m.get_field(f)
            assert np.linalg.norm(a - got) <= 1e-7 * np.linalg.norm(a), (m.spec.nx, f)
    b.close()
    for c in alone + mixed:
        c.close()
