"""Systems of unequal masses in physical units: with lengths of 1e13 to 1e16 and
masses of 1e30, as in SI or CGS, 1 / r^3 is below the float range where m / r^3
is well inside it.  The single-precision modes form the latter without the
former: accelerations and the velocity change of a step against the oracle, at
each mode's own bar.  One size per path: small systems' steps in one kernel
(480), separate kernels (3000), the two-pass mixed mode (13000)."""
import ctypes as C
import math

import numpy as np
import pytest

from paper_1003_3896_gb300 import ics

pytestmark = pytest.mark.gpu

TOL = {"ds": 1e-6, "ds_full": 1e-6, "ds_near": 1e-6, "fp32": 1e-4}


@pytest.fixture(scope="module")
def nbs():
    from paper_1003_3896_gb300 import build
    build.build()
    from paper_1003_3896_gb300 import nbsym
    return nbsym


def rel_rms(a, ref):
    return math.sqrt(((a - ref) ** 2).sum() / (ref ** 2).sum())


def system(n, length, mass):
    """A Plummer sphere of unequal masses, G = 1, lengths and masses scaled."""
    pos, vel, m = ics.plummer(n, 4, masses=ics.salpeter_masses(n, 4))
    m = m / m.mean() * mass
    vel = vel * math.sqrt(m.sum() / length)
    return pos * length, vel, m, 0.01 * length


@pytest.mark.parametrize("length,mass", [(1e13, 1e30), (1e15, 1e30), (1e16, 2e33), (1e-12, 1e-6)])
@pytest.mark.parametrize("n", [480, 3000, 13000])
@pytest.mark.parametrize("prec", list(TOL))
def test_unequal_masses_in_physical_units(nbs, orc, prec, n, length, mass):
    pos, vel, m, eps = system(n, length, mass)
    ref = orc.accel_int(pos, m, 1.0, eps)
    dt = 1e-3 * math.sqrt(length ** 3 / m.sum())
    p = orc.Params(G=1.0, eps=eps)
    with nbs.Context(n, eps=eps, precision=prec) as c:
        c.load(pos, vel, m)
        assert rel_rms(c.accel(), ref) <= TOL[prec]
        c.step(2, dt, 1)
        _, v = c.get_state()
    _, want = orc.run(pos, vel, m, p, 2, dt, 1)
    assert rel_rms(v - vel, want - vel) <= TOL[prec]


@pytest.mark.parametrize("equal", [False, True])
@pytest.mark.parametrize("prec", list(TOL))
def test_static_entry_point_in_physical_units(nbs, orc, prec, equal):
    """nb_accel_static takes the general-mass form for equal masses too."""
    torch = pytest.importorskip("torch")
    n = 3000
    pos, _, m, eps = system(n, 1e15, 1e30)
    if equal:
        m = np.full(n, 1e30)
    tp, tm = torch.from_numpy(pos).cuda(), torch.from_numpy(m).cuda()
    out = torch.empty((n, 3), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    p = nbs.Params()
    nbs.nb_params_default(C.byref(p))
    p.precision = nbs.PRECISIONS[prec]
    p.eps = eps
    rc = nbs.nb_accel_static(C.byref(p), n, tp.data_ptr(), tm.data_ptr(), out.data_ptr())
    assert rc == nbs.NB_OK, nbs.nb_last_error()
    torch.cuda.synchronize()
    assert rel_rms(out.cpu().numpy(), orc.accel_int(pos, m, 1.0, eps)) <= TOL[prec]
