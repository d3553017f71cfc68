"""The scalars of the FP64 one-barrier CG in integer arithmetic (csrc/pcg_scalar.cuh), checked on
the host against exact rationals: alpha and beta of the single-reduction recurrence.  The
arithmetic carries 57 bits or more, so beta is within one unit of FP64's last place and alpha
within the two roundings of delta - beta^2 den_old, at the conditioning of that difference."""
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
    src = os.path.join(ROOT, "tests", "native", "cg_scalars_host.cu")
    subprocess.check_call([build._nvcc(), "-std=c++17", "-O2", "-Xcompiler", "-fPIC", "-shared", "-I",
                           os.path.join(ROOT, "include"), "-I", CSRC, "-o", so, src])
    L = ctypes.CDLL(so)
    dp = ctypes.POINTER(ctypes.c_double)
    L.sch_step.argtypes = [ctypes.c_double] * 4 + [dp, dp]
    L.sch_step.restype = None
    L.sch_digits.argtypes = [ctypes.POINTER(ctypes.c_longlong), ctypes.c_int]
    L.sch_digits.restype = ctypes.c_double
    return L


def _step(lib, *a):
    al, be = ctypes.c_double(np.nan), ctypes.c_double(np.nan)
    lib.sch_step(*a, ctypes.byref(al), ctypes.byref(be))
    return al.value, be.value


def _draws():
    rng = np.random.default_rng(4)
    for k in range(3000):
        g0 = float(rng.uniform(1, 2) * 2.0 ** rng.integers(-300, 300))
        g1 = g0 * float(rng.uniform(1, 2) * 2.0 ** rng.integers(-12, 12))
        d0 = g0 * float(rng.uniform(1, 2) * 2.0 ** rng.integers(-3, 6))
        t = (g1 / g0) ** 2 * d0
        # the difference keeps between all and 2^-30 of delta's bits, or is negative
        delta = t * (1 + float(rng.uniform(1, 2) * 2.0 ** -int(rng.integers(-6, 30)))) if k % 10 else t * float(rng.uniform(0.1, 0.9))
        yield g0, d0, g1, delta
    for m in (1.0, 2.0 - 2.0 ** -52, 1.5):  # significands at the ends of their range
        for n in (1.0, 2.0 - 2.0 ** -52):
            yield m, n, n, 4 * m
            yield m, m, n, 8 * n


def test_alpha_and_beta_against_exact_rationals(lib):
    for g0, d0, g1, delta in _draws():
        alpha, beta = _step(lib, g0, d0, g1, delta)
        G0, D0, G1, D = map(Fraction, (g0, d0, g1, delta))
        B = G1 / G0
        den = D - B * B * D0
        assert abs(Fraction(beta) / B - 1) <= Fraction(1, 2 ** 52)
        cond = abs(D / den) + 1
        assert abs(Fraction(alpha) * den / G1 - 1) <= cond * Fraction(1, 2 ** 52)


def test_zero_denominator_keeps_alpha(lib):
    al, be = ctypes.c_double(7.0), ctypes.c_double(0.0)
    lib.sch_step(1.0, 3.0, 2.0, 12.0, ctypes.byref(al), ctypes.byref(be))  # delta = beta^2 den_old
    assert al.value == 7.0 and be.value == 2.0


@pytest.mark.parametrize("digits", [[0, 0, 0, 0, 0], [1, 0, 0, 0, 0], [-5, 7, 0, 0, 0], [2 ** 35, -2 ** 35, 2 ** 35, 3, 1],
                                    [-1, -1, -1, -1, -1], [0, 0, 0, 0, 2 ** 21]])
def test_digit_sums_round_once(lib, digits):
    S = (ctypes.c_longlong * 5)(*digits)
    exact = sum(Fraction(d) * 2 ** (26 * k) for k, d in enumerate(digits))
    got = Fraction(lib.sch_digits(S, -100)) * 2 ** 100
    assert abs(got - exact) <= abs(exact) * Fraction(1, 2 ** 53)
