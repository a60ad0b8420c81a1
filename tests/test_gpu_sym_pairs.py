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


MIXED_SIZES = SIZES + [1, 2, 63, 191, 1024, 1281, 2049, 4097]


@pytest.mark.parametrize("n", MIXED_SIZES)
def test_two_pass_mixed_form(nbs, orc, n):
    """The mixed mode's float pairs (chunks of 64 j bodies, rows of 64 to 256 i
    bodies) with the near-pair pass, at the mixed bar 1e-6; eps = 0 takes the
    self-masked own rows."""
    for equal, eps in ((True, 0.01), (False, 0.01), (False, 0.0)):
        pos, vel, m = bodies(n, equal)
        with nbs.Context(n, eps=eps, precision="ds_near") as c:
            c.load(pos, vel, m)
            a = c.accel()
            np.testing.assert_array_equal(c.accel(), a)
        if n == 1:
            assert np.all(a == 0)
            continue
        ref = orc.accel_int(pos, m, 1.0, eps)
        assert rel_rms(a, ref) <= 1e-6, (equal, eps, rel_rms(a, ref))


@pytest.mark.parametrize("n,pairs", [(1500, 1), (12001, 20), (16384, 64), (12001, 1500)])
def test_bodies_in_close_encounters(nbs, orc, n, pairs):
    """A Plummer sphere in which `pairs` pairs of bodies are close binaries: each
    partner pulls its body far harder than the cluster does, so the bodies are
    summed apart, or, past their limit (the last case), not.  Every body of a
    binary and 200 others at the per-body bar 5e-6 of the two-pass form (error
    over the acceleration, at least a tenth of the rms), twice bit for bit."""
    pos, vel, m = ics.plummer(n, 5)
    rng = np.random.default_rng(pairs)
    pick = rng.permutation(n)[:2 * pairs].reshape(-1, 2)
    sep = 0.05 / math.sqrt(n)
    u = rng.normal(size=(pairs, 3))
    pos[pick[:, 1]] = pos[pick[:, 0]] + sep * u / np.linalg.norm(u, axis=1)[:, None]
    eps = ics.paper_softening(n)
    with nbs.Context(n, eps=eps, precision="ds_near") as c:
        c.load(pos, vel, m)
        a = c.accel()
        np.testing.assert_array_equal(c.accel(), a)
    idx = np.unique(np.concatenate([pick.ravel()[:400], rng.choice(n, 200, replace=False)]))
    ref = orc.accel_int_at(pos, m, idx, 1.0, eps)
    size = np.linalg.norm(ref, axis=1)
    other = np.setdiff1d(idx, pick.ravel())
    floor = 0.1 * math.sqrt((orc.accel_int_at(pos, m, other, 1.0, eps) ** 2).sum(1).mean())
    err = np.linalg.norm(a[idx] - ref, axis=1) / np.maximum(size, floor)
    assert err.max() <= 5e-6, err.max()
