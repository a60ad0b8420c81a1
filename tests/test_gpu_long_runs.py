"""Graphs of 16 steps (from 96 steps at one length on) and half drifts shared by
neighbouring steps give the bits of the same steps one call at a time: in mixed
precision with every pair in double-single, in float-float and in double precision,
with the full and with the symmetric kernels, at the run lengths where the kinds of
graph meet, in one call and in calls that reach the length together."""
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


@pytest.mark.parametrize("prec,n", [("ds", 1500), ("fp32", 1500), ("fp64", 300), ("fp64", 1024),
                                    ("dd", 700), ("dd", 1300)])
def test_long_runs_equal_single_steps(nbs, prec, n):
    pos, vel, m = ics.plummer(n, 3)
    pos, vel = ics.place_on_orbit(pos, vel)

    def run(calls):
        with nbs.Context(n, eps=1e-2, precision=prec, ext_on=True) as c:
            c.load(pos, vel, m)
            for k in calls:
                c.step(2, 1 / 512, k)
            return c.get_state()

    want = {}
    for calls in ([96], [112], [113], [31, 64, 18], [64, 49], [48, 48, 17]):
        t = sum(calls)
        if t not in want:
            want[t] = run([1] * t)   # one step a graph, no drift shared
        got = run(calls)
        for q in range(2):
            np.testing.assert_array_equal(got[q], want[t][q], err_msg=str(calls))
