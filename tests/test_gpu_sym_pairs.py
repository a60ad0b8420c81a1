"""The symmetric pair kernels (each unordered pair once, its force added to both
bodies) at the sizes where they can go wrong: one warp's row, a block's rows
full, one short and one over, ragged last blocks, odd and even block counts
(the half-distance tile belongs to one row only), unequal masses (the two sides'
scales differ), and the unsoftened self term; against the oracle at the
FP64-class bar 1e-12 of the other parity tests (relative RMS), and sum m a = 0
to the rounding of its terms."""
import math

import numpy as np
import pytest

from paper_1003_3896_gb300 import ics

pytestmark = pytest.mark.gpu

SIZES = [3, 31, 32, 33, 65, 127, 129, 255, 256, 257, 383, 385, 511, 513, 640, 769, 1025, 1537,
         2560, 7000]


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


@pytest.mark.parametrize("prec", ["fp64", "dd"])
@pytest.mark.parametrize("n", SIZES)
def test_accel_and_energy(nbs, orc, prec, n):
    for equal, eps in ((True, 0.01), (False, 0.01), (False, 0.0)):
        pos, vel, m = bodies(n, equal)
        ref = orc.accel_int(pos, m, 1.0, eps)
        want = orc.energy(pos, vel, m, orc.Params(eps=eps))
        with nbs.Context(n, eps=eps, precision=prec) as c:
            c.load(pos, vel, m)
            a = c.accel()
            e = c.energy()
        assert rel_rms(a, ref) <= 1e-12, (equal, eps, rel_rms(a, ref))
        f = m[:, None] * a
        assert np.abs(f.sum(0)).max() <= 1e-12 * np.abs(f).sum(), (equal, eps)
        assert abs(e.W - want.W) <= 1e-12 * abs(want.W), (equal, eps)


@pytest.mark.parametrize("prec", ["fp64", "dd"])
def test_uneven_clusters_of_both_mass_kinds(nbs, orc, prec):
    """Clusters around the block width in one launch, some of equal and some
    of unequal masses, and more clusters than travel by value."""
    for sizes in (SIZES, [1, 2, 33, 130, 300] * 120):
        cl = [bodies(n, k % 2 == 0) for k, n in enumerate(sizes)]
        pos, vel, m = (np.concatenate([c[q] for c in cl]) for q in range(3))
        with nbs.Context(sizes=sizes, precision=prec, eps=0.01) as b:
            b.load(pos, vel, m)
            a = b.accel()
            e = b.energy_clusters()
        off = 0
        for k, n in enumerate(sizes):
            if k < 20 and n > 1:
                ref = orc.accel_int(cl[k][0], cl[k][2], 1.0, 0.01)
                assert rel_rms(a[off:off + n], ref) <= 1e-12, (k, n)
                want = orc.energy(*cl[k], orc.Params(eps=0.01))
                assert abs(e[k].W - want.W) <= 1e-12 * abs(want.W), (k, n)
            off += n
