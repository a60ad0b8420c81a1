"""Bodies in a close encounter are summed apart (near_encounter_kernel): in an order
that does not depend on the shape of the pair kernel's launch.  So between two
shapes of the symmetric kernel their accelerations keep every bit, where those of
the other bodies, whose float partial sums are cut elsewhere, do not; and above the
number of such bodies that are looked after, theirs do not either."""
import math

import numpy as np
import pytest

from paper_1003_3896_gb300 import ics

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nbs():
    from paper_1003_3896_gb300 import build
    build.build()
    from paper_1003_3896_gb300 import nbsym
    yield nbsym
    nbsym.tune_clear()


@pytest.mark.parametrize("equal", [True, False])
@pytest.mark.parametrize("n,pairs,kept", [(12001, 20, True), (16384, 64, True), (16384, 1500, False)])
def test_encounter_sums_do_not_depend_on_the_shape(nbs, tmp_path, n, pairs, kept, equal):
    pos, vel, m = ics.plummer(n, 5, masses=None if equal else ics.salpeter_masses(n, n))
    rng = np.random.default_rng(pairs)
    pick = rng.permutation(n)[:2 * pairs].reshape(-1, 2)
    u = rng.normal(size=(pairs, 3))
    pos[pick[:, 1]] = pos[pick[:, 0]] + 0.02 / math.sqrt(n) * u / np.linalg.norm(u, axis=1)[:, None]
    # the heavier partner's pull decides: the lighter body of each pair
    light = np.where(m[pick[:, 0]] <= m[pick[:, 1]], pick[:, 0], pick[:, 1])
    eps = ics.paper_softening(n)
    nbs.tune_clear()
    with nbs.Context(n, eps=eps, precision="ds") as c:
        c.load(pos, vel, m)
        c.tune(1)
    path = tmp_path / "shapes.txt"
    nbs.tune_save(str(path))
    head, entry = path.read_text().split("\n")[:2]
    got = []
    for bodies in (4, 8):
        f = entry.split()
        f[5] = str(bodies)   # sms precision K n size: then the bodies per thread
        path.write_text(head + "\n" + " ".join(f) + "\n")
        nbs.tune_clear()
        assert nbs.tune_load(str(path)) == 1
        with nbs.Context(n, eps=eps, precision="ds") as c:
            c.load(pos, vel, m)
            assert c.pair_symmetric and c.pair_shape()["bodies_per_thread"] == bodies
            got.append(c.accel())
    nbs.tune_clear()
    same = (got[0] == got[1]).all(axis=1)
    other = np.setdiff1d(np.arange(n), pick.ravel())
    assert same[other].mean() < 0.9
    if kept:
        assert same[light].all()
    else:
        assert same[light].mean() < 0.9
