"""Sums below FP64's normal range in the one-barrier FP64 solve: the integer scalars (csrc/pcg_scalar.cuh)
round to subnormal numbers like FP64 does, so that a solve with a tiny right-hand side runs to its tolerance
instead of taking a residual norm that underflows for zero."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2211_10698_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2211_10698_gb300 import build

    so = str(tmp_path_factory.mktemp("sch") / "libsch.so")
    subprocess.check_call([build._nvcc(), "-std=c++17", "-O2", "-Xcompiler", "-fPIC", "-shared", "-I",
                           os.path.join(ROOT, "include"), "-I", CSRC, "-o", so,
                           os.path.join(ROOT, "tests", "native", "cg_scalars_host.cu")])
    L = ctypes.CDLL(so)
    L.sch_digits.argtypes = [ctypes.POINTER(ctypes.c_longlong), ctypes.c_int]
    L.sch_digits.restype = ctypes.c_double
    return L


def test_rounding_down_to_the_smallest_subnormal(lib):
    rng = np.random.default_rng(2)
    values = [1, 2, 3, 2 ** 52, 2 ** 53 - 1, 2 ** 53 + 1, 2 ** 63, 2 ** 63 + 1, 2 ** 64 - 1]
    values += [int(rng.integers(1, 2 ** 62)) for _ in range(300)]
    for v in values:
        for sign in (1, -1):
            digits = (ctypes.c_longlong * 5)(*[sign * ((v >> (26 * k)) & (2 ** 26 - 1)) for k in range(5)])
            n = v.bit_length()
            for top in range(-1080, -1015, 3):  # the value's power of two, through the end of the range
                lo = top - n
                want = float(Fraction(sign * v) * Fraction(2) ** lo)  # correctly rounded
                assert lib.sch_digits(digits, lo) == want, (v, lo)


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny", [(128, 64), (300, 150)])
def test_tiny_right_hand_side(orc, nx, ny):
    """||b||^2 about 1e-290, so that the squared residual at the tolerance is about 1e-310; the cells' own
    squares keep three digits and more there."""
    from paper_2211_10698_gb300 import ccm, inputs as I

    c = I.make_case("tiny", nx, ny, (-2.0, 6.0, -2.0, 2.0), I.Geometry(kind=I.GEOM_CIRCLE, cx=0.1, cy=-0.05, r=0.5), re=100.0,
                    cfl=0.5, lref=1.0)
    c.tol_p, c.autotune = 1e-10, 0
    o = orc.Oracle(c)
    b = np.random.default_rng(0).standard_normal(c.shape) * o.active
    g = ccm.Case(c)
    plain = g.solve_pressure(b)
    g.set_field(ccm.CCM_F_PHI, np.zeros(c.shape))
    tiny = b * (1e-145 / np.linalg.norm(b))
    st = g.solve_pressure(tiny)
    assert plain["converged"] and st["converged"]
    assert abs(st["iters"] - plain["iters"]) <= 0.02 * plain["iters"] + 2, (st, plain)
    r = (tiny - o.poisson(g.get_field(ccm.CCM_F_PHI)))[o.active]
    assert np.linalg.norm(r / 1e-145) <= 1.1e-10
    g.close()
