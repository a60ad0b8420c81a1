"""Steps of a small system in one kernel give the bits of the separate kernels
(which a profiled context runs), at the edges of the blocks' shares of the
bodies, of the frame's segments and of the path's range."""
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


@pytest.mark.parametrize("prec", ["ds", "fp32"])
@pytest.mark.parametrize("n", [1, 2, 15, 17, 64, 255, 480, 511, 513, 777, 1023, 1024, 1025])
def test_small_steps_equal_separate_kernels(nbs, n, prec):
    pos, vel, m = ics.plummer(n, n)
    for order, eps, ext, spec in [(2, 0.0, False, False), (6, 1e-2, True, True),
                                  (2, 1e-3, True, False)]:
        mm = m * (1 + np.arange(n) % 5) if spec else m
        p, v = ics.place_on_orbit(pos, vel) if ext else (pos, vel)

        def run(prof, calls):
            with nbs.Context(n, eps=eps, precision=prec, ext_on=ext) as c:
                c.load(p, v, mm)
                c.prof_enable(prof)
                for k in calls:
                    c.step(order, 1 / 512, k)
                return c.get_state()

        a, b, one = run(False, [7]), run(True, [7]), run(False, [1, 5, 1])
        for q in range(2):
            np.testing.assert_array_equal(a[q], b[q])
            np.testing.assert_array_equal(a[q], one[q])
