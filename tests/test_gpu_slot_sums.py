"""Adding up a body's partial sums with one, two, four or eight warps per 32
bodies: the accelerations against plain 64-bit sums, and the kick against the
accelerations, on both sides of the sizes where the number changes."""
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


# Per unit of sum |m d / r^3|: fp64 and dd the worst case of a sum of 4096 terms in
# a row (2^-53 each; a run of a slot is shorter); ds 16 roundings to 24 bits.
TOL = {"fp64": 4096 * 2.0 ** -53, "dd": 4096 * 2.0 ** -53, "ds": 16 * 2.0 ** -24}


@pytest.mark.parametrize("prec", ["fp64", "dd", "ds"])
@pytest.mark.parametrize("n", [513, 2587, 14592, 14593, 29184, 29185, 58368, 58369])
def test_slot_sums(nbs, n, prec):
    pos, vel, m = ics.plummer(n, 11)
    eps, dt = 1e-2, 1.0 / 1024
    with nbs.Context(n, eps=eps, precision=prec) as c:
        c.load(pos + 0.5 * dt * vel, vel, m)
        a = c.accel()
    with nbs.Context(n, eps=eps, precision=prec) as c:
        c.load(pos, vel, m)
        c.step(2, dt, 1)
        kicked = c.get_state()[1]
    x = pos + 0.5 * dt * vel
    pick = np.unique(np.concatenate([np.arange(0, n, n // 40), [0, 31, 32, n - 1]]))
    for i in pick:
        d = x - x[i]
        w = m / (np.einsum("ij,ij->i", d, d) + eps * eps) ** 1.5
        exact = w @ d
        size = float(w @ np.sqrt(np.einsum("ij,ij->i", d, d)))
        assert np.abs(a[i] - exact).max() <= TOL[prec] * size
        assert np.abs((kicked[i] - vel[i]) / dt - exact).max() <= TOL[prec] * size + 2.0 ** -51 / dt
