"""Cases of different sizes solved from two threads at once: the launches of one thread ask for more
shared memory than the other's, on the same kernel, and neither may see the other's limit."""
import threading

import numpy as np
import pytest

from paper_2211_10698_gb300 import ccm, inputs as I

pytestmark = pytest.mark.gpu


STILL = ((I.BC_DIRICHLET, I.BC_OUTFLOW, I.BC_OUTFLOW, I.BC_OUTFLOW), (0.0,) * 4, (0.0,) * 4)


def _case(nx, ny, precision, degree, plan):
    """A fluid at rest, so that two iterations are enough for its steps."""
    c = I.make_case("thread", nx, ny, (-2.0, 6.0, -2.0, 2.0), I.Geometry(kind=I.GEOM_CIRCLE, cx=0.1, cy=-0.05, r=0.5), re=100.0,
                    cfl=0.5, lref=1.0, bc=STILL)
    c.precision, c.autotune, c.max_iter_p = precision, 0, 2
    c.precond, c.cheb_degree = ("chebyshev", degree) if degree > 1 else ("jacobi", 1)
    g = ccm.Case(c)
    if plan:
        g.set_launch_plan(plan)
    return g


def _together(*jobs):
    errors = []

    def loop(job):
        try:
            for _ in range(1500):
                job()
        except Exception as e:
            errors.append(e)

    ts = [threading.Thread(target=loop, args=(j,)) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors[:1]


# (precision, degree, a larger case and its plan, a smaller one on the same kernel and its plan)
PAIRS = [("fp64", 1, (400, 200, None), (300, 150, None)),                               # resident tiles, built-in
         ("mixed", 3, (128, 64, None), (61, 37, None)),                                 # band tiles, built-in
         ("fp64", 1, (128, 64, (0, 0, 0, 0, 0, 8, 0)), (61, 37, (0, 0, 0, 0, 0, 8, 0))),  # cluster
         ("mixed", 3, (128, 64, (64, 16, 2, 8, 0, 0, 1)), (61, 37, (32, 8, 2, 10, 0, 0, 1)))]


@pytest.mark.parametrize("precision,degree,large,small", PAIRS)
def test_solves_from_two_threads(precision, degree, large, small):
    cases = [_case(s[0], s[1], precision, degree, s[2]) for s in (large, small)]
    rhs = [np.random.default_rng(k).standard_normal(c.shape) for k, c in enumerate(cases)]
    _together(*[lambda c=c, b=b: c.solve_pressure(b) for c, b in zip(cases, rhs)])
    for c in cases:
        c.close()


def test_batches_from_two_threads():
    jobs = []
    for sizes in ([(256, 128), (128, 64)], [(61, 37), (40, 24)]):
        b = ccm.Batch(len(sizes))
        for s in sizes:
            b.add(_case(*s, "fp64", 1, None))
        b.set_tuning(False)
        b.set_graphs(False)
        jobs.append(lambda b=b: b.step(1))
    _together(*jobs)
