"""A pool whose caller leaves the launch shape open, around the number of runs
where it changes its block size, and the read-back of physical positions
through free arena space: in one piece, in several, and without any."""
import math

import numpy as np
import pytest

import paper_1108_1954_gb300 as pic
import torch  # noqa: F401
import workloads as W

pytestmark = pytest.mark.gpu
L = 4.0 * math.pi


def state(n, seed):
    return W.to_f32_state(*W.two_stream(n, L, 0.2, 0.02, seed), L)


@pytest.mark.parametrize("runs", [1, 37, 38, 39, 90])
def test_open_shape_equals_alone(runs):
    ps = [pic.Params(npart=2000 + 37 * i, ncell=1 + (53 * i) % 2048, length=L) for i in range(runs)]
    pool = pic.Pool(max_slots=runs, ncell_max=2048, arena_bytes=1 << 26, history=16,
                    device="cuda:0")
    slots = [pool.admit(p, *state(p.npart, i), 6) for i, p in enumerate(ps)]
    pool.advance(6)
    for i in (0, runs // 2, runs - 1):
        run = pic.Run(ps[i], device="cuda:0")
        run.init(*state(ps[i].npart, i))
        run.step_n(6)
        for a, b in zip(pool.get_cells(slots[i]), run.get_cells()):
            assert np.array_equal(a, b)
        assert np.array_equal(pool.get_field(slots[i])["rho_q"], run.get_field()["rho_q"])


@pytest.mark.parametrize("n,free", [(250001, 1 << 20), (250001, 300 << 10), (250001, 0),
                                    (1001, 4352), (1001, 0), (1, 0)])
def test_positions_read_back_through_free_space(n, free):
    p = pic.Params(npart=n, ncell=300, length=L)
    table = 1 << 14
    pool = pic.Pool(max_slots=4, ncell_max=512, arena_bytes=table + pic.pool_run_bytes(p, 16) + free,
                    history=16, device="cuda:0")
    # fill what the table leaves beyond `free` with a second run's particles
    slot = pool.admit(p, *state(n, 3), 2)
    pool.advance(2)
    used, idle = pool.usage()
    spare = idle - free
    small = pic.Params(npart=1, ncell=1, length=L)
    while spare >= pic.pool_run_bytes(small, 16) and pool.admit(small, *state(1, 1), 0) is not None:
        spare = pool.usage()[1] - free
    u, v = pool.get_cells(slot)
    want = np.minimum((u.astype(np.float64) * (L / 300)).astype(np.float32),
                      np.nextafter(np.float32(L), np.float32(0)))
    x, w = pool.get_state(slot)
    assert np.array_equal(x, want) and np.array_equal(w, v)
    xt = torch.empty(n, pin_memory=True)
    vt = torch.empty(n, pin_memory=True)
    pool.get_state(slot, xt, vt)
    assert np.array_equal(xt.numpy(), want) and np.array_equal(vt.numpy(), v)


def alone(p, seed, steps):
    run = pic.Run(p, device="cuda:0")
    run.init(*state(p.npart, seed))
    run.step_n(steps)
    return run


@pytest.mark.parametrize("variant,cluster,block,ncell_max",
                         [(1, 8, 256, 2048), (2, 8, 256, 2048), (5, 4, 512, 2048), (6, 2, 512, 1024),
                          (1 + 16, 8, 256, 2048), (5 + 16, 8, 512, 4096), (6 + 16, 1, 512, 512)])
def test_many_runs_keep_the_cluster_launch(variant, cluster, block, ncell_max):
    # more runs than there are SMs: no many-step launch, whatever their sizes
    n = 160
    ps = [pic.Params(npart=1000 + 61 * i, ncell=1 + (97 * i) % ncell_max, length=L) for i in range(n)]
    pool = pic.Pool(max_slots=n, ncell_max=ncell_max, arena_bytes=1 << 27, history=16, variant=variant,
                    cluster=cluster, block=block, device="cuda:0")
    slots = [pool.admit(p, *state(p.npart, i), 5) for i, p in enumerate(ps)]
    pool.advance(2)
    pool.advance(3)
    for i in (0, 1, n // 2, n - 1):
        run = alone(ps[i], i, 5)
        for a, b in zip(pool.get_cells(slots[i]), run.get_cells()):
            assert np.array_equal(a, b)
        f, g = pool.get_field(slots[i]), run.get_field()
        assert np.array_equal(f["rho_q"], g["rho_q"]) and np.array_equal(f["E"], g["E"])


@pytest.mark.parametrize("free", [8 << 20, 0])
def test_few_uneven_runs_equal_alone(free):
    # the many-step launch, and without room for its accumulators the clusters;
    # runs that stop early, one- and two-cell grids, the largest NG it takes
    specs = [(600001, 4096, 9, 0), (3, 1, 9, 0), (5, 2, 4, 0), (40000, 1025, 9, 0), (70001, 64, 1, 0),
             (20003, 2049, 7, 50), (20003, 333, 9, 3)]
    ps = [pic.Params(npart=n, ncell=g, length=L, sort_interval=S) for n, g, _, S in specs]
    pool = pic.Pool(max_slots=len(ps), ncell_max=4096, variant=5, cluster=8, block=512, history=16,
                    arena_bytes=(1 << 14) + sum(pic.pool_run_bytes(p, 16) for p in ps) + free,
                    device="cuda:0")
    slots = [pool.admit(p, *state(p.npart, i), k) for i, (p, (_, _, k, _)) in enumerate(zip(ps, specs))]
    assert None not in slots
    for k in (1, 2, 1, 9):             # the last run sorts before steps 3 and 6
        pool.advance(k)
    for i, (p, (_, _, k, _)) in enumerate(zip(ps, specs)):
        assert pool.step_count(slots[i]) == k
        run = alone(p, i, k)
        for a, b in zip(pool.get_cells(slots[i]), run.get_cells()):
            assert np.array_equal(a, b)
        f, g = pool.get_field(slots[i]), run.get_field()
        for key in ("rho_q", "E", "rho"):
            assert np.array_equal(f[key], g[key])
        d, e = pool.diagnostics(slots[i], 0, k + 1), run.diagnostics(0, k + 1)
        assert np.array_equal(d["step"], e["step"]) and np.array_equal(d["charge_q"], e["charge_q"])
        np.testing.assert_allclose(d["field"], e["field"], rtol=1e-12, atol=1e-300)
        np.testing.assert_allclose(d["kinetic"][:-1], e["kinetic"][:-1], rtol=1e-5)
        assert np.isnan(d["kinetic"][-1])


def two_kernels(p, seed, steps):
    """The run alone by push and solve kernels (a shape of its own)."""
    q = pic.Params(npart=p.npart, ncell=p.ncell, length=L, sort_interval=p.sort_interval, block_size=256)
    return alone(q, seed, steps)


def assert_equal_runs(pool, slot, run):
    for a, b in zip(pool.get_cells(slot), run.get_cells()):
        assert np.array_equal(a, b)
    f, g = pool.get_field(slot), run.get_field()
    for key in ("rho_q", "E", "rho"):
        assert np.array_equal(f[key], g[key])


def many_step_launched(pool):
    """Whether an advance takes the many-step launch: its waits are made to run out."""
    pool.set_wait_limit(4096, 1)
    try:
        pool.advance(1)
        return False
    except pic.PicError as e:
        assert e.code == pic.PIC_ETIMEOUT
        return True
    finally:
        pool.set_wait_limit()


@pytest.mark.parametrize("how,many", [("open", True), ("config", False), ("block", False), ("configured", False),
                                      ("allowed", True), ("forbidden", False)])
def test_a_chosen_shape_is_taken(how, many):
    kw = dict(config=dict(variant=5, cluster=2, block=512), allowed=dict(variant=5, cluster=2, block=512),
              block=dict(block=256)).get(how, {})
    pool = pic.Pool(max_slots=1, ncell_max=64, arena_bytes=1 << 24, history=16, device="cuda:0", **kw)
    if how == "configured":
        pool.configure(17, 4, 256)
    elif how in ("allowed", "forbidden"):
        pool.many_step(how == "allowed")
    p = pic.Params(npart=20000, ncell=64, length=L)
    slot = pool.admit(p, *state(20000, 1), 5)
    pool.advance(2)
    assert many_step_launched(pool) == many
    if not many:
        pool.advance(2)
        assert_equal_runs(pool, slot, two_kernels(p, 1, 5))


@pytest.mark.parametrize("variant,cluster,block,ncell_max",
                         [(2, 8, 256, 2048), (1, 8, 256, 2048), (5, 4, 512, 2048), (2, 2, 512, 1024), (2, 1, 512, 512),
                          (1, 4, 256, 1024), (2 + 16, 8, 512, 4096), (5 + 16, 8, 256, 2048)])
def test_chosen_shapes_equal_the_two_kernels(variant, cluster, block, ncell_max):
    sizes = [(20000, 64), (100003, 2048), (5, 16), (1, 1), (77777, 512), (250001, 1024), (65537, 4096)]
    ps = [pic.Params(npart=n, ncell=g, length=L) for n, g in sizes if g <= ncell_max]
    pool = pic.Pool(max_slots=len(ps), ncell_max=ncell_max, arena_bytes=1 << 27, history=32, variant=variant,
                    cluster=cluster, block=block, device="cuda:0")
    slots = [pool.admit(p, *state(p.npart, i), 12) for i, p in enumerate(ps)]
    pool.advance(5)
    pool.advance(7)
    for i, p in enumerate(ps):
        assert_equal_runs(pool, slots[i], two_kernels(p, i, 12))


@pytest.mark.parametrize("runs", [1, 37, 38, 39, 90])
def test_open_clusters_on_both_sides_of_the_block_size_equal_the_two_kernels(runs):
    # blocks of 512 threads while every run has a cluster of its own, then of 256
    ps = [pic.Params(npart=2000 + 37 * i, ncell=1 + (53 * i) % 2048, length=L) for i in range(runs)]
    pool = pic.Pool(max_slots=runs, ncell_max=2048, arena_bytes=1 << 26, history=16, device="cuda:0")
    pool.many_step(False)
    slots = [pool.admit(p, *state(p.npart, i), 6) for i, p in enumerate(ps)]
    pool.advance(6)
    for i in (0, runs // 2, runs - 1):
        assert_equal_runs(pool, slots[i], two_kernels(ps[i], i, 6))


def test_many_step_runs_of_a_pool_equal_the_two_kernels():
    specs = [(600001, 2048, 9, 0), (3, 1, 9, 0), (5, 2, 4, 0), (40000, 1025, 9, 0), (70001, 64, 1, 0), (20003, 1024, 7, 50)]
    ps = [pic.Params(npart=n, ncell=g, length=L, sort_interval=S) for n, g, _, S in specs]
    pool = pic.Pool(max_slots=len(ps), ncell_max=2048, history=16, arena_bytes=1 << 26, device="cuda:0")
    slots = [pool.admit(p, *state(p.npart, i), k) for i, (p, (_, _, k, _)) in enumerate(zip(ps, specs))]
    for k in (1, 2, 1, 9):
        pool.advance(k)
    for i, (p, (_, _, k, _)) in enumerate(zip(ps, specs)):
        assert pool.step_count(slots[i]) == k
        assert_equal_runs(pool, slots[i], two_kernels(p, i, k))
    pool.release(slots[0])
    pool.admit(ps[1], *state(3, 1), 5)
    assert many_step_launched(pool)


def test_read_backs_from_several_threads_beside_admissions():
    # the threads' conversions share the arena's idle space, which an admission takes from
    import threading
    sizes = [300007, 200003, 90001, 50021]
    ps = [pic.Params(npart=n, ncell=300, length=L) for n in sizes]
    extra = pic.Params(npart=70001, ncell=100, length=L)
    need = (1 << 14) + sum(pic.pool_run_bytes(p, 16) for p in ps) + pic.pool_run_bytes(extra, 16)
    pool = pic.Pool(max_slots=8, ncell_max=512, arena_bytes=need + (600 << 10), history=16, device="cuda:0")
    slots = [pool.admit(p, *state(p.npart, i), 3) for i, p in enumerate(ps)]
    pool.advance(3)
    want = [pool.get_state(s) for s in slots]
    x, v = state(extra.npart, 9)
    errors = []

    def read(i):
        try:
            for _ in range(40):
                a, b = pool.get_state(slots[i])
                assert np.array_equal(a, want[i][0]) and np.array_equal(b, want[i][1])
                assert np.array_equal(pool.get_field(slots[i])["rho_q"], fields[i])
        except BaseException as e:
            errors.append(e)

    fields = [pool.get_field(s)["rho_q"] for s in slots]
    threads = [threading.Thread(target=read, args=(i,)) for i in range(len(ps))]
    [t.start() for t in threads]
    for _ in range(20):
        s = pool.admit(extra, x, v, 1)
        pool.release(s)
    s = pool.admit(extra, x, v, 2)
    [t.join() for t in threads]
    assert not errors, errors[0]
    pool.advance(2)
    assert_equal_runs(pool, s, two_kernels_of(extra, x, v, 2))


def two_kernels_of(p, x, v, steps):
    run = pic.Run(pic.Params(npart=p.npart, ncell=p.ncell, length=L, block_size=256), device="cuda:0")
    run.init(x, v)
    run.step_n(steps)
    return run
