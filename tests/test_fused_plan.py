"""Tile plans of the one-barrier FP64 solve (csrc/fused_plan.h), on the CPU: every grid that the
allocation-free solve takes has a resident plan within its fixed scratch, and the mailboxes that a case
carves hold every resident plan that a caller can set."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2211_10698_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("plan") / "libplan.so")
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                           "-o", so, os.path.join(ROOT, "tests", "native", "fused_plan_host.cpp")])
    L = ctypes.CDLL(so)
    L.check_noalloc.restype = L.mail_excess.restype = L.noalloc_max_elems.restype = ctypes.c_long
    L.check_noalloc.argtypes = [ctypes.c_int, ctypes.c_long, ctypes.POINTER(ctypes.c_int)]
    L.plan_of.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_long, ctypes.POINTER(ctypes.c_int)]
    return L


# the 152 SMs of the whole part and the least this family is sold with; 227 KB less a block's static part
@pytest.mark.parametrize("sms", [152, 148, 132])
def test_every_grid_of_the_allocation_free_solve_has_a_plan(lib, sms):
    bad = (ctypes.c_int * 3)()
    n = lib.check_noalloc(sms, 227 * 1024 - 20 * 1024, bad)
    assert list(bad) == [0, 0, 0] and n > 500_000


def test_a_limit_on_the_mailboxes_changes_no_plan_that_meets_it(lib):
    rng = np.random.default_rng(0)
    for _ in range(2000):
        nx, ny = (int(np.exp(rng.uniform(np.log(4), np.log(4000)))) for _ in range(2))
        free, held = (ctypes.c_int * 4)(), (ctypes.c_int * 4)()
        lib.plan_of(nx, ny, 152, -1, free)
        need = 4 * free[3] * (free[1] + min(free[0], nx))
        lib.plan_of(nx, ny, 152, need, held)
        if free[3]:
            assert 4 * held[3] * (held[1] + min(held[0], nx)) <= need
            # (another width may take fewer, taller tiles under the limit; never smaller ones)
            assert held[1] * min(held[0], nx) == free[1] * min(free[0], nx)


def test_a_cases_mailboxes_hold_every_resident_plan(lib):
    rng = np.random.default_rng(1)
    for _ in range(400):
        nx, ny = (int(np.exp(rng.uniform(np.log(4), np.log(4000)))) for _ in range(2))
        for tx in (32, 64, 128, 256, 512):
            for ty in range(1, ny + 1):
                assert lib.mail_excess(nx, ny, tx, ty) <= 0, (nx, ny, tx, ty)
