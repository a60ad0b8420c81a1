"""A call of several steps (graphs of 16 steps, half drifts shared by
neighbouring steps in double precision) gives the bits of the same steps one
call at a time, at the run lengths where the kinds of graph meet."""
import numpy as np
import pytest

from paper_1003_3896_gb300 import ics

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nbs():
    from paper_1003_3896_gb300 import build
    build.build()
    from paper_1003_3896_gb300 import nbsym
    return nbsym


@pytest.mark.parametrize("prec", ["fp64", "ds", "dd"])
@pytest.mark.parametrize("order", [2, 6])
def test_runs_of_steps_equal_single_steps(nbs, prec, order):
    n = 300
    pos, vel, m = ics.plummer(n, 3)
    pos, vel = ics.place_on_orbit(pos, vel)

    def run(calls):
        with nbs.Context(n, eps=1e-2, precision=prec, ext_on=True) as c:
            c.load(pos, vel, m)
            for k in calls:
                c.step(order, 1 / 512, k)
            return c.get_state()

    for total in (2, 15, 16, 17, 32, 33, 49):
        x, v = run([total])
        x1, v1 = run([1] * total)
        np.testing.assert_array_equal(x, x1)
        np.testing.assert_array_equal(v, v1)
    x, v = run([50])
    x1, v1 = run([16, 1, 33])
    np.testing.assert_array_equal(x, x1)
    np.testing.assert_array_equal(v, v1)
