"""Performance cases of the direct-summation N-body library: what its users
have it do, through the Python binding of the C ABI.

Each case is one call pattern of a simulation program: advance a resident
system (``Context.step``) and read its state, evaluate accelerations once,
read the energy diagnostic, or hand a batch of integration jobs to the serving
loop.  Sizes, softenings and step lengths are those of the repository's
benchmark workloads, the paper's test workload, and odd sizes between them.

``prepare`` makes seeded synthetic inputs and the context (or server) a
program keeps; ``run`` is one pass; ``exact`` restates the method in plain
64-bit torch for the same inputs.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1003_3896_gb300 import ics

#: Largest pair count N^2 x evaluations of a drawn case: the largest listed
#: one's (a single evaluation of 262144 bodies).
MAX_PAIRS = 262144 ** 2

#: Kick weights of the sixth-order scheme (Yoshida's solution A).
W1, W2, W3 = -1.17767998417887, 0.235573213359357, 0.784513610477560
SI6A = (W3, W2, W1, 1.0 - 2.0 * (W1 + W2 + W3), W1, W2, W3)


def listed():
    return [
        # The paper's smallest system (Table 3, N = 480): one leapfrog step per
        # call, the loop of a program that looks at the state after each step.
        # Launches and host latency are what counts.
        dict(name="sphere_480_ds_step", kind="step", model="sphere", n=480, prec="ds", order=2,
             dt=5e-4, steps=1, eps=0.0, field=False, mbh=0.0),
        # 1024 bodies in double precision, 64 leapfrog steps, state read back
        # to the host: a small high-accuracy run.
        dict(name="henon_1024_fp64_64steps", kind="step", model="henon", n=1024, prec="fp64",
             order=2, dt=1.0 / 1024, steps=64, eps=1e-3, field=False, mbh=0.0, host=True),
        # The paper's middle size in pure single precision, one leapfrog step.
        dict(name="sphere_30720_fp32_step", kind="step", model="sphere", n=30720, prec="fp32",
             order=2, dt=5e-4, steps=1, eps=0.0, field=False, mbh=0.0),
        # A cluster falling through a galactic centre with a massive black
        # hole, mixed precision, sixth order: a few steps between outputs.
        dict(name="plunge_15360_ds_si6a", kind="step", model="plunge", n=15360, prec="ds", order=6,
             dt=2e-4, steps=4, eps=0.0, field=True, mbh=1.0),
        # The headline workload: a 65536-body cluster on an orbit in the disk +
        # bulge field, mixed precision, one sixth-order step.
        dict(name="orbit_65536_ds_si6a", kind="step", model="orbit", n=65536, prec="ds", order=6,
             dt=1.0 / 256, steps=1, eps=0.0, field=True, mbh=0.0),
        # The largest: one mixed-precision force evaluation of 262144 bodies
        # with a mass spectrum.
        dict(name="salpeter_262144_ds_accel", kind="accel", model="salpeter", n=262144, prec="ds",
             eps=1e-4),
        # FP64-class accelerations on the single-precision pipes, odd size,
        # mass spectrum.
        dict(name="salpeter_50021_dd_accel", kind="accel", model="salpeter", n=50021, prec="dd",
             eps=1e-4),
        # The plain double-precision evaluation.
        dict(name="plummer_16384_fp64_accel", kind="accel", model="plummer", n=16384, prec="fp64",
             eps=0.0),
        # 512 independent clusters of 256 to 8192 bodies, mixed precision, one
        # sixth-order step of all of them.
        dict(name="ensemble_512_ds_si6a", kind="ensemble", clusters=512, lo=256, hi=8192, sizes=0,
             prec="ds", order=6, dt=1.0 / 512, steps=1),
        # A few dozen small ragged clusters in float-float, four leapfrog steps.
        dict(name="ensemble_48_small_dd", kind="ensemble", clusters=48, lo=100, hi=1500, sizes=3,
             prec="dd", order=2, dt=1.0 / 1024, steps=4),
        # Energy, momentum and angular momentum of a 32768-body system between
        # stretches of integration.
        dict(name="energy_32768", kind="energy", model="orbit", n=32768, eps=0.0, field=True),
        # The serving loop: eight queued jobs of mixed size, order and
        # precision, host arrays in and out.
        dict(name="serve_8_jobs", kind="serve", jobs=8, lo=1024, hi=20000, mix=1),
    ]


def _log_int(rng, lo, hi):
    """Log-uniform integer on [lo, hi]."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "accel", "accel", "ensemble", "ensemble", "energy",
                       "serve"])
    if kind == "step":
        prec = rng.choice(["ds", "ds", "fp32", "dd", "fp64"])
        order = rng.choice([2, 6])
        model = rng.choice(["sphere", "henon", "orbit", "plunge"])
        hi = {"ds": 90000, "fp32": 90000, "dd": 40000, "fp64": 12000}[prec]
        n = _log_int(rng, 256, hi)
        steps = max(1, min(rng.choice([1, 2, 4, 16]),
                           MAX_PAIRS // (n * n * (7 if order == 6 else 1) * 2)))
        return dict(kind=kind, model=model, n=n, prec=prec, order=order,
                    dt={"sphere": 5e-4, "henon": 1.0 / 1024, "orbit": 1.0 / 256,
                        "plunge": 2e-4}[model],
                    steps=steps, eps=0.0, field=model in ("orbit", "plunge"),
                    mbh=rng.choice([0.1, 1.0, 50.0]) if model == "plunge" else 0.0)
    if kind == "accel":
        prec = rng.choice(["ds", "ds_full", "fp32", "dd", "fp64"])
        hi = {"ds": 250000, "ds_full": 200000, "fp32": 250000, "dd": 80000, "fp64": 25000}[prec]
        return dict(kind=kind, model=rng.choice(["plummer", "salpeter", "sphere"]),
                    n=_log_int(rng, 256, hi), prec=prec, eps=rng.choice([0.0, 1e-4, 1e-2]))
    if kind == "ensemble":
        hi = _log_int(rng, 600, 8192)
        return dict(kind=kind, clusters=_log_int(rng, 2, 512), lo=rng.choice([100, 256]), hi=hi,
                    sizes=rng.randrange(1000), prec=rng.choice(["ds", "ds", "fp32", "dd"]),
                    order=rng.choice([2, 6]), dt=1.0 / 1024, steps=1)
    if kind == "energy":
        return dict(kind=kind, model=rng.choice(["orbit", "plunge"]), n=_log_int(rng, 256, 40000),
                    eps=0.0, field=True)
    return dict(kind=kind, jobs=rng.randrange(2, 12), lo=512, hi=_log_int(rng, 4000, 20000),
                mix=rng.randrange(1000))


# ---- inputs ----------------------------------------------------------------

def _bodies(case, seed):
    """(positions, velocities, masses, softening) of a one-cluster case."""
    n, model = case["n"], case["model"]
    if model == "sphere":
        pos, vel, m = ics.uniform_sphere(n, seed)
    elif model == "henon":
        pos, vel, m = ics.henon_plummer(n, seed)
    elif model == "salpeter":
        pos, vel, m = ics.plummer(n, seed, masses=ics.salpeter_masses(n, seed))
    elif model == "plunge":
        pos, vel, m = ics.plunge_cluster(n, seed)
    else:
        pos, vel, m = ics.plummer(n, seed)
        if model == "orbit":
            pos, vel = ics.place_on_orbit(pos, vel)
    return pos, vel, m, case["eps"] or ics.paper_softening(n)


def _clusters(case, seed):
    """[(positions, velocities, masses, softening)] of an ensemble case."""
    sizes = ics.ensemble_sizes(case["clusters"], case["lo"], case["hi"], seed=case["sizes"])
    return [(*ics.henon_plummer(int(n), seed * 1024 + k), ics.paper_softening(int(n)))
            for k, n in enumerate(sizes)]


def _jobs(case, seed):
    """The serving case's jobs: sizes log-uniform, order 2 or 6, double or
    mixed precision, step counts that keep the whole batch at some tens of
    milliseconds of GPU work."""
    rng = np.random.default_rng(case["mix"])
    jobs = []
    for k in range(case["jobs"]):
        n = int(round(math.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"])))))
        order = int(rng.choice([2, 6]))
        prec = str(rng.choice(["fp64", "ds"]))
        pairs = n * n * (7 if order == 6 else 1)
        steps = int(max(2, min(40, 2e9 / pairs)))
        pos, vel, m = ics.henon_plummer(n, seed * 64 + k)
        jobs.append(dict(pos=pos, vel=vel, mass=m, order=order, prec=prec, steps=steps,
                         dt=1.0 / 1024, eps=ics.paper_softening(n)))
    return jobs


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# ---- one pass --------------------------------------------------------------

def prepare(case, seed):
    from paper_1003_3896_gb300 import nbsym
    if case["kind"] == "serve":
        return dict(case=case, jobs=_jobs(case, seed), server=nbsym.Server())
    if case["kind"] == "ensemble":
        cl = _clusters(case, seed)
        ctx = nbsym.Context(sizes=[c[2].size for c in cl], precision=case["prec"])
        ctx.set_cluster_params(eps=[c[3] for c in cl])
        pos, vel, m = (np.concatenate([c[q] for c in cl]) for q in range(3))
    else:
        pos, vel, m, eps = _bodies(case, seed)
        ctx = nbsym.Context(m.size, eps=eps, precision=case.get("prec", "ds"),
                            ext_on=case.get("field", False), Mbh=case.get("mbh", 0.0),
                            eps_bh=0.05)
    p, v, mm = _gpu(pos), _gpu(vel), _gpu(m)
    torch.cuda.synchronize()
    ctx.load_device(m.size, p, v, mm)
    return dict(case=case, ctx=ctx, a=torch.empty_like(p), b=torch.empty_like(p))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "serve":
        srv = state["server"]
        ids = [srv.submit(j["pos"], j["vel"], j["mass"], j["order"], j["dt"], j["steps"],
                          precision=j["prec"], eps=j["eps"]) for j in state["jobs"]]
        for i in ids:
            srv.wait(i)
        out = [srv.result(i) for i in ids]
        for i in ids:
            srv.forget(i)
        return out
    ctx = state["ctx"]
    if kind == "energy":
        e = ctx.energy()
        return dict(K=e.K, W=e.W, W_ext=e.W_ext, E=e.E, P=e.P, L=e.L)
    if kind == "accel":
        ctx.accel_device(state["a"])
        # the single-precision modes' accelerations are handed on as the
        # single-precision numbers that they are good to
        return state["a"] if case["prec"] in ("fp64", "dd") else state["a"].float()
    ctx.step(case["order"], case["dt"], case["steps"])
    if case.get("host"):
        return ctx.get_state()
    ctx.get_state_device(state["a"], state["b"])
    return state["a"], state["b"]


def work(case):
    """The least one pass can do: each unordered pair once at 24 flops (three
    differences, r^2 + eps^2, the inverse square root and its cube, both
    bodies' three sums), the state read and written once."""
    kind = case["kind"]
    if kind == "serve":
        rng = np.random.default_rng(case["mix"])
        pairs = bodies = 0
        for _ in range(case["jobs"]):
            n = int(round(math.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"])))))
            order = int(rng.choice([2, 6]))
            rng.choice(["fp64", "ds"])
            one = n * n * (7 if order == 6 else 1)
            pairs += one * int(max(2, min(40, 2e9 / one)))
            bodies += n
    else:
        if kind == "ensemble":
            sizes = ics.ensemble_sizes(case["clusters"], case["lo"], case["hi"],
                                       seed=case["sizes"])
            bodies, pairs = int(sizes.sum()), int((sizes ** 2).sum())
        else:
            bodies, pairs = case["n"], case["n"] ** 2
        if kind in ("step", "ensemble"):
            pairs *= case["steps"] * (7 if case["order"] == 6 else 1)
    return {"bytes": 104.0 * bodies, "flops": 12.0 * pairs}


# ---- the same in plain 64-bit torch ----------------------------------------

def _rsqrt3(r2):
    return 1.0 / (r2 * torch.sqrt(r2))


def _pair_accel(x, m, eps):
    n = x.shape[0]
    out = torch.empty_like(x)
    rows = max(1, (1 << 25) // n)
    for i in range(0, n, rows):
        d = [x[None, :, c] - x[i:i + rows, None, c] for c in range(3)]
        w = m * _rsqrt3(d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps * eps)
        for c in range(3):
            out[i:i + rows, c] = (w * d[c]).sum(1)
    return out


def _pair_potential(x, m, eps):
    n = x.shape[0]
    out = torch.empty(n, dtype=x.dtype, device=x.device)
    rows = max(1, (1 << 25) // n)
    for i in range(0, n, rows):
        r2 = sum((x[None, :, c] - x[i:i + rows, None, c]) ** 2 for c in range(3)) + eps * eps
        w = m / torch.sqrt(r2)
        k = torch.arange(i, min(n, i + rows), device=x.device)
        w[k - i, k] = 0.0
        out[i:i + rows] = w.sum(1)
    return out


MD, AD, BD, MB, AB = ics.DISK_BULGE
EPS_BH = 0.05


def _field_accel(x, mbh):
    R2 = x[:, 0] ** 2 + x[:, 1] ** 2
    zb = torch.sqrt(x[:, 2] ** 2 + BD * BD)
    kd = MD * _rsqrt3(R2 + (AD + zb) ** 2)
    k = MB * _rsqrt3(R2 + x[:, 2] ** 2 + AB * AB)
    if mbh > 0:
        k = k + mbh * _rsqrt3(R2 + x[:, 2] ** 2 + EPS_BH * EPS_BH)
    return -torch.stack([(kd + k) * x[:, 0], (kd + k) * x[:, 1],
                         (kd * (AD + zb) / zb + k) * x[:, 2]], 1)


def _integrate(x, v, m, eps, order, dt, steps, field=False, mbh=0.0):
    for _ in range(steps):
        for w in (1.0,) if order == 2 else SI6A:
            x = x + (0.5 * w * dt) * v
            a = _pair_accel(x, m, eps)
            if field:
                a = a + _field_accel(x, mbh)
            v = v + (w * dt) * a
            x = x + (0.5 * w * dt) * v
    return x, v


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        out = []
        for j in _jobs(case, seed):
            x, v = _integrate(_gpu(j["pos"]), _gpu(j["vel"]), _gpu(j["mass"]), j["eps"],
                              j["order"], j["dt"], j["steps"])
            out.append((x.cpu().numpy(), v.cpu().numpy()))
        return out
    if kind == "ensemble":
        got = [_integrate(_gpu(p), _gpu(v), _gpu(m), e, case["order"], case["dt"], case["steps"])
               for p, v, m, e in _clusters(case, seed)]
        return torch.cat([g[0] for g in got]), torch.cat([g[1] for g in got])
    pos, vel, m, eps = _bodies(case, seed)
    x, v, m = _gpu(pos), _gpu(vel), _gpu(m)
    if kind == "accel":
        return _pair_accel(x, m, eps)
    if kind == "energy":
        R2 = x[:, 0] ** 2 + x[:, 1] ** 2
        r2 = R2 + x[:, 2] ** 2
        phi = (-MD / torch.sqrt(R2 + (AD + torch.sqrt(x[:, 2] ** 2 + BD * BD)) ** 2)
               - MB / torch.sqrt(r2 + AB * AB))
        K = float(0.5 * (m * (v * v).sum(1)).sum())
        W = float(-0.5 * (m * _pair_potential(x, m, eps)).sum())
        We = float((m * phi).sum()) if case["field"] else 0.0
        return dict(K=K, W=W, W_ext=We, E=K + W + We, P=(m[:, None] * v).sum(0).cpu().numpy(),
                    L=(m[:, None] * torch.linalg.cross(x, v)).sum(0).cpu().numpy())
    x, v = _integrate(x, v, m, eps, case["order"], case["dt"], case["steps"], case["field"],
                      case["mbh"])
    return (x.cpu().numpy(), v.cpu().numpy()) if case.get("host") else (x, v)
