"""The symmetric pair kernels at sizes that take them (small systems keep the full
kernels; test_host_plans.py checks that each size here is on the right side of the
line): ragged last blocks, odd and even block counts, both mass forms, clusters by
value and from the device tables.  And the two float-float kernels on the same
bodies: a system gives the same sums whichever kernel it takes."""
import math

import numpy as np
import pytest

from paper_1003_3896_gb300 import ics

pytestmark = pytest.mark.gpu

SINGLE = [("fp64", n) for n in (785, 895, 896, 897, 1151, 1281, 2049)] + \
         [("dd", n) for n in (1201, 1279, 1281, 1409, 1792, 2047, 6145)] + \
         [("ds_near", n) for n in (11586, 11647, 12033, 12289, 18433)]
CLUSTERS = [("fp64", [1, 33, 130, 300] * 20), ("fp64", [1, 2, 33, 130, 300] * 120),
            ("dd", [1, 33, 129, 257, 640, 1281, 2560]), ("dd", [1, 257, 300, 385, 513] * 120)]
TOL = {"fp64": 1e-12, "dd": 1e-12, "ds_near": 1e-6}


@pytest.fixture(scope="module")
def nbs():
    from paper_1003_3896_gb300 import build
    build.build()
    from paper_1003_3896_gb300 import nbsym
    return nbsym


def bodies(n, equal):
    return ics.plummer(n, 70 + n, masses=None if equal else ics.salpeter_masses(n, n))


def rel_rms(a, ref):
    return math.sqrt(((a - ref) ** 2).sum() / (ref ** 2).sum())


@pytest.mark.parametrize("prec,n", SINGLE)
def test_one_system(nbs, orc, prec, n):
    for equal, eps in ((True, 0.01), (False, 0.01), (False, 0.0)):
        pos, vel, m = bodies(n, equal)
        with nbs.Context(n, eps=eps, precision=prec) as c:
            c.load(pos, vel, m)
            assert c.pair_symmetric
            a = c.accel()
        assert rel_rms(a, orc.accel_int(pos, m, 1.0, eps)) <= TOL[prec], (equal, eps)


@pytest.mark.parametrize("prec,sizes", CLUSTERS, ids=lambda v: v if isinstance(v, str) else len(v))
def test_clusters(nbs, orc, prec, sizes):
    cl = [bodies(n, k % 2 == 0) for k, n in enumerate(sizes)]
    pos, vel, m = (np.concatenate([c[q] for c in cl]) for q in range(3))
    with nbs.Context(sizes=sizes, precision=prec, eps=0.01) as b:
        b.load(pos, vel, m)
        assert b.pair_symmetric
        a = b.accel()
    off = np.concatenate([[0], np.cumsum(sizes)])
    for k in [*range(min(20, len(sizes))), len(sizes) - 1]:
        if sizes[k] > 1:
            ref = orc.accel_int(cl[k][0], cl[k][2], 1.0, 0.01)
            assert rel_rms(a[off[k]:off[k + 1]], ref) <= TOL[prec], k


@pytest.mark.parametrize("equal", [True, False])
@pytest.mark.parametrize("n", [2, 33, 65, 129, 161, 256, 257, 300, 385, 513, 777, 1024])
def test_float_float_sums_do_not_depend_on_the_kernel(nbs, n, equal):
    """Alone (the full kernel) and beside a 4100-body cluster (the symmetric one):
    a body's sums over 32 others have the same terms in the same order, so what is
    left are the double additions of its at most n / 32 + 40 partial sums and slots,
    2^-53 each of the running sum, at random: 2e-15 at most."""
    for seed in (1, 2, 3):
        cl = [ics.plummer(q, seed * 100 + q, masses=None if equal else ics.salpeter_masses(q, q))
              for q in (n, 4100)]
        pos, vel, m = (np.concatenate([c[q] for c in cl]) for q in range(3))
        with nbs.Context(sizes=[n, 4100], precision="dd", eps=1e-3) as b:
            b.load(pos, vel, m)
            assert b.pair_symmetric
            got = b.accel()[:n]
        with nbs.Context(n, precision="dd", eps=1e-3) as c:
            c.load(*cl[0])
            assert not c.pair_symmetric
            alone = c.accel()
            parts = np.concatenate([c.accel_range(0, n // 2), c.accel_range(n // 2, n)])
        assert rel_rms(got, alone) <= 2e-15
        assert rel_rms(parts, alone) <= 2e-15
