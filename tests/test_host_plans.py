"""What a context does when a plan cannot get its device memory, on a stand-in
for the CUDA runtime (hostcuda.py): no captured graph outlives the memory it was
captured with, a context whose plan failed goes on with the plan it had or, where
that fails too, refuses every call that would launch until a plan succeeds."""
import numpy as np
import pytest

from hostcuda import Host
from paper_1003_3896_gb300 import ics

N = 40000   # the double-precision plan's partial sums outgrow those of the others


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    return Host(tmp_path_factory.mktemp("hostcuda"))


@pytest.fixture()
def ctx(host):
    host.fail_from()
    c = host.nbsym.Context(N, eps=1e-2, precision="fp32")
    c.load(*ics.plummer(N, 1))
    host.clear()
    yield c
    host.fail_from()
    c.close()


def refused(host, f):
    """f() is NB_ESTATE before any launch."""
    host.clear()
    with pytest.raises(host.nbsym.NBError) as e:
        f()
    assert e.value.code == host.nbsym.NB_ESTATE
    assert not host.launches() and host.graphs == 0


def test_graphs_do_not_outlive_the_storage(host, ctx):
    """A change of precision that moves the partial sums, with and without room."""
    ctx.step(2, 1e-3, 1)
    ctx.set_precision("fp64")
    ctx.step(2, 1e-3, 1)
    ctx.set_precision("fp32")
    ctx.step(2, 1e-3, 1)
    assert host.stale == 0
    ctx.set_precision("ds")
    ctx.step(6, 1e-3, 2)
    assert host.stale == 0 and host.ran("pair_sym")


def test_no_room_for_symmetric_slots_takes_the_full_kernels(host, ctx):
    host.fail_from(80 << 20)   # the full kernels' 69 MB still fit
    ctx.set_precision("fp64")
    ctx.step(2, 1e-3, 1)
    assert host.ran("pair_fp64_kernelILi1E") and not host.ran("pair_sym")
    assert host.stale == 0


@pytest.mark.parametrize("prec,n,kernel", [("dd", 440000, "pair_ff_kernelILi1E"),
                                           ("fp64", 320000, "pair_fp64_kernelILi1E")])
def test_slots_beyond_the_limit_take_the_full_kernels_shape(host, prec, n, kernel):
    """More than the 4 GB that symmetric slots may take."""
    host.fail_from()
    with host.nbsym.Context(n, eps=1e-2, precision=prec) as c:
        c.load(np.zeros((n, 3)), np.zeros((n, 3)), np.ones(n))
        host.clear()
        c.accel()
        assert host.ran(kernel) and not host.ran("pair_sym")


@pytest.mark.parametrize("change", ["precision", "load", "params"])
def test_failed_plan_leaves_a_usable_or_refusing_context(host, ctx, change):
    nb = host.nbsym
    if change == "load":
        ctx.load(*ics.plummer(N // 4, 1))   # small sums, to outgrow
    ctx.step(2, 1e-3, 1)

    def again():
        if change == "precision":
            ctx.set_precision("fp64")
        elif change == "load":
            ctx.set_precision("fp64")
            ctx.load(*ics.plummer(N, 1))
        else:
            ctx.set_precision("fp64")
            ctx.set_cluster_params(eps=[1e-3])

    host.fail_from(1 << 20)
    with pytest.raises(nb.NBError) as e:
        again()
    assert e.value.code == nb.NB_ENOMEM
    out = np.empty((ctx.n, 3))
    for f in (lambda: ctx.step(2, 1e-3, 1), ctx.accel, ctx.energy, ctx.get_state, ctx.torque,
              lambda: ctx.set_state(pos=out), lambda: ctx.tune(1), ctx.accel_symmetric,
              lambda: ctx.accel_range(0, 10), lambda: ctx.substep_range(0, 10, 0.1, 0.1)):
        refused(host, f)
    host.fail_from()
    again()
    host.clear()
    ctx.step(2, 1e-3, 1)
    assert host.ran("pair_sym_kernel") and host.stale == 0


def test_failed_load_keeps_the_old_system(host):
    """Room for what the context has (5000 bodies: 15 MB of partial sums), none for
    what it asks for."""
    nb = host.nbsym
    with nb.Context(N, eps=1e-2, precision="fp32") as c:
        c.load(*ics.plummer(5000, 1))
        c.step(2, 1e-3, 1)
        shape = c.pair_shape()
        host.clear()
        host.fail_from(20 << 20)
        try:
            with pytest.raises(nb.NBError) as e:
                c.load(*ics.plummer(N, 1))
            assert e.value.code == nb.NB_ENOMEM
            assert c.n == 5000 and c.pair_shape() == shape
            c.step(2, 1e-3, 1)
            assert host.graphs == 1 and host.stale == 0
        finally:
            host.fail_from()


@pytest.mark.parametrize("prec,n,kernel,ipb", [
    ("dd", 65536, "pair_ff_kernelILi1E", 256), ("dd", 5000, "pair_ff_kernelILi1E", 256),
    ("fp64", 32768, "pair_fp64_kernelILi1E", 128), ("fp64", 700, "pair_fp64_kernelILi1E", 128),
    ("ds_near", 15360, "pair_sp_kernelILi2E", 512), ("ds_near", 65536, "pair_sp_kernelILi4E", 1024),
    ("fp32", 65536, "pair_sp_kernelILi4E", 1024)])
def test_range_launches_take_the_full_kernels_shape(host, prec, n, kernel, ipb):
    """An eighth of the bodies: a block per i-block row of the full kernel's own
    width, not of the symmetric plan's."""
    host.fail_from()
    with host.nbsym.Context(n, eps=1e-2, precision=prec) as c:
        c.load(*ics.plummer(n, 1))
        for f in (lambda: c.accel_range(0, n // 8), lambda: c.substep_range(0, n // 8, 0.1, 0.1)):
            host.clear()
            f()
            assert [k[1] for k in host.ran(kernel)] == [-(-(n // 8) // ipb)]
            assert not host.ran("pair_sym")


def test_no_room_for_the_encounter_sums_takes_the_full_kernels(host, ctx):
    """The partial sums are there (they serve every precision), 1 MB more is not."""
    host.fail_from(100 << 10)
    ctx.set_precision("ds")
    ctx.step(2, 1e-3, 1)
    assert host.ran("pair_sp_kernel") and not host.ran("pair_sym") and not host.ran("encounter")
    host.fail_from()
    ctx.set_precision("ds")
    host.clear()
    ctx.step(2, 1e-3, 1)
    assert host.ran("pair_sym") and host.ran("encounter") and host.stale == 0


def test_serving_groups_grow_without_stopping_the_device(host):
    """Jobs of growing size in the mixed mode's large groups: neither cudaMalloc nor
    cudaFree, which wait for every group's work, once the server stands."""
    host.fail_from()
    nb = host.nbsym
    with nb.Server(hbm_budget_bytes=1e8) as srv:
        host.clear()
        for n in (12000, 20000, 30000, 40000):
            pos, vel, m = ics.plummer(n, 1)
            jid = srv.submit(pos, vel, m, 6, 1e-3, 2, precision="ds", eps=1e-2)
            assert srv.wait(jid, 60)["state"] == nb.JOB_DONE
        assert len(host.ran("encounter")) == 4 * 2 * 7
        assert host.syncing == 0


def _server_growth(host, jobs, **kw):
    """Device bytes that a server of the default budget takes for these jobs."""
    nb = host.nbsym
    with nb.Server(hbm_budget_bytes=4e9, **kw) as srv:
        host.clear()
        start = host.live
        for n, order, prec in jobs:
            pos, vel, m = ics.plummer(n, 1)
            jid = srv.submit(pos, vel, m, order, 1e-3, 1, precision=prec, eps=1e-2)
            assert srv.wait(jid, 60)["state"] == nb.JOB_DONE
        return host.live - start, bool(host.ran("pair_sym_kernel"))


def test_server_partial_sums_stay_within_the_groups_allowance(host):
    """Large jobs of every group: the symmetric slots of 65536 bodies take 119 MB where
    the allowance of unused groups covers them, else what is left; in all at most
    67 MB for each of the twelve groups and 48 bytes per body of each."""
    host.fail_from()
    n = 65536
    grown, sym = _server_growth(host, [(n, 6, "ds")])
    assert sym and grown <= 140e6
    # all groups may have jobs: no group beyond its own 67 MB
    grown, _ = _server_growth(host, [(n, 6, "ds")], fp64_via_dd=0)
    assert grown <= 67e6 + 60 * n
    jobs = [(m, order, prec) for m in (4000, n, 2 * n) for order in (2, 6) for prec in ("ds", "dd")]
    grown, _ = _server_growth(host, jobs)
    assert grown <= 12 * 67e6 + 60 * sum(j[0] for j in jobs)


def test_server_takes_little_at_creation_with_a_small_budget(host):
    """What creation takes beyond its share per budget byte."""
    host.fail_from()
    live = []
    for budget in (1e8, 2e8):
        before = host.live
        with host.nbsym.Server(hbm_budget_bytes=budget):
            live.append(host.live - before)
    assert 2 * live[0] - live[1] <= 8e6
    before = host.live
    with host.nbsym.Server(hbm_budget_bytes=4e9, max_jobs=4):
        pass
    assert host.live == before


def _chosen(host, prec, sizes):
    host.fail_from()
    kw = dict(capacity=sizes[0]) if len(sizes) == 1 else dict(sizes=sizes)
    with host.nbsym.Context(eps=1e-2, precision=prec, **kw) as c:
        n = sum(sizes)
        c.load(np.zeros((n, 3)), np.zeros((n, 3)), np.ones(n))
        host.clear()
        c.accel()
        assert c.pair_symmetric == bool(host.ran("pair_sym"))
        return c.pair_symmetric


def test_sizes_of_the_symmetric_kernels_tests_take_them(host):
    import test_gpu_sym_sizes as t
    for prec, n in t.SINGLE:
        assert _chosen(host, prec, [n]), (prec, n)
    for prec, sizes in t.CLUSTERS:
        assert _chosen(host, prec, sizes), (prec, len(sizes))


@pytest.mark.parametrize("prec,sizes,sym", [
    ("dd", [64], False), ("dd", [700], False), ("dd", [1200], False), ("dd", [1201], True),
    ("dd", [400, 700], False), ("dd", [450] * 12, False), ("dd", [450] * 100, True),
    ("dd", [100] * 1000, False), ("dd", [300, 4100], True), ("fp64", [784], False),
    ("fp64", [785], True), ("ds_near", [11585], False), ("ds_near", [11586], True), ("ds", [11586], True),
    ("ds_near", [20000, 3], False), ("fp32", [40000], False), ("ds_full", [40000], False)])
def test_which_sets_take_the_symmetric_kernels(host, prec, sizes, sym):
    """Both sides of the lines drawn in use_sym, where each side measured faster."""
    assert _chosen(host, prec, sizes) == sym


def test_new_step_lengths_capture_one_small_graph_each(host):
    """A program that changes dt at every call; one that keeps it; several in turn."""
    host.fail_from()
    for prec, n in (("fp64", 300), ("fp64", 1024), ("ds", 2000), ("dd", 2000)):
        with host.nbsym.Context(n, eps=1e-2, precision=prec) as c:
            c.load(*ics.plummer(n, 1))
            for order, steps in ((2, 2), (2, 16), (2, 17), (6, 1), (6, 4)):
                host.clear()
                for k in range(5):
                    c.step(order, 1e-3 * (1 + k + 10 * steps), steps)
                assert host.captures == 5 and host.graphs == 5 * steps
            # kept: from 96 steps on in graphs of 16
            host.clear()
            c.step(2, 1e-4, 64)
            assert host.graphs == 64
            host.clear()
            c.step(2, 1e-4, 64)
            assert host.graphs == 4
            host.clear()
            c.step(2, 1e-4, 64)
            assert host.graphs == 4 and host.captures == 0
            host.clear()
            c.step(2, 2e-4, 100)
            assert host.graphs == 6 + 4
            # eight lengths in turn: captured for good
            for r in range(6):
                if r == 5:
                    host.clear()
                for k in range(8):
                    c.step(2, 3e-4 * (1 + k), 33)
            assert host.captures == 0


@pytest.mark.parametrize("prec", ["ds", "fp64"])
def test_tuning_gives_its_partial_sums_back(host, prec):
    """The candidates reach the narrowest i-blocks' slots; what stays is what the chosen
    shape takes in a fresh context."""
    host.fail_from()
    n = 60000
    nb = host.nbsym
    body = ics.plummer(n, 1)
    before = host.live
    try:
        with nb.Context(n, eps=1e-2, precision=prec) as c:
            c.load(*body)
            c.step(2, 1e-3, 1)
            host.clear()
            c.tune(1)
            shape, held = c.pair_shape(), host.live - before
            assert host.peak - before > 1.5 * held
            c.step(2, 1e-3, 1)
            assert host.stale == 0
        with nb.Context(n, eps=1e-2, precision=prec) as c:   # takes the tuned shape
            c.load(*body)
            assert c.pair_shape() == shape
            assert host.live - before == held
    finally:
        nb.tune_clear()


@pytest.mark.parametrize("n", [520000, 530000, 600000, 700000])
def test_symmetric_mixed_plans_look_for_encounters(host, n):
    """Also near the size where the symmetric slots no longer fit."""
    host.fail_from()
    with host.nbsym.Context(n, eps=1e-2, precision="ds") as c:
        c.load(np.zeros((n, 3)), np.zeros((n, 3)), np.ones(n))
        host.clear()
        c.accel()
        assert bool(host.ran("pair_sym")) == bool(host.ran("encounter"))
        assert bool(host.ran("pair_sym")) == (n <= 600000)


def test_pair_symmetric_without_a_plan(host):
    host.fail_from()
    nb = host.nbsym
    assert nb.nb_pair_symmetric(None) == nb.NB_EINVAL
    with nb.Context(10) as c, pytest.raises(nb.NBError) as e:
        c.pair_symmetric
    assert e.value.code == nb.NB_ESTATE


@pytest.mark.parametrize("prec,n,order,one", [
    ("ds", 1, 2, True), ("ds", 480, 2, True), ("ds", 1024, 2, True), ("ds", 1025, 2, False),
    ("ds", 704, 6, True), ("ds", 705, 6, False), ("fp32", 832, 6, True), ("fp32", 833, 6, False),
    ("fp64", 480, 2, False), ("dd", 480, 2, False), ("ds_near", 480, 2, False)])
def test_which_steps_run_in_one_kernel(host, prec, n, order, one):
    """The sizes of the small-step tests that compare it with the separate kernels take
    it, and a profiled context, the other side of that comparison, does not."""
    host.fail_from()
    with host.nbsym.Context(n, eps=1e-2, precision=prec) as c:
        c.load(*ics.plummer(n, 1))
        host.clear()
        c.step(order, 1e-3, 3)
        assert bool(host.ran("small_step_kernel")) == one
        assert host.graphs == (0 if one else 3)
        c.prof_enable(True)
        host.clear()
        c.step(order, 1e-3, 3)
        assert not host.ran("small_step_kernel") and host.graphs == 3


@pytest.mark.parametrize("prec", ["ds", "fp64", "dd"])
def test_first_load_reserves_once(host, prec):
    """The plan before the masses are known takes no less than the one after: no large
    storage is freed and allocated again."""
    host.fail_from()
    with host.nbsym.Context(N, eps=1e-2, precision=prec) as c:
        host.clear()
        c.load(*ics.plummer(N, 1))
        assert host.syncing <= 2   # partial sums, encounter sums
