"""The many-step launch (a run whose launch shape is left open) against the
push and solve kernels, which an explicit shape selects: the particles, the
density, E and the histories' exact entries bit for bit, whatever the sizes
and however the steps are split into calls."""
import math

import numpy as np
import pytest

import paper_1108_1954_gb300 as pic
import torch  # noqa: F401

pytestmark = pytest.mark.gpu
L = 4.0 * math.pi


def state(n, seed):
    rng = np.random.default_rng(seed)
    x = rng.uniform(0.0, L, n).astype(np.float32)
    x[x >= np.float32(L)] = 0.0
    if n > 2:
        x[0], x[1] = 0.0, np.nextafter(np.float32(L), np.float32(0))
    return x, rng.normal(0.0, 0.4, n).astype(np.float32)


def pair(n, ng, **kw):
    a = pic.Run(pic.Params(npart=n, ncell=ng, length=L, **kw), device="cuda:0")
    # an explicit block size (NGP: its one variant) keeps the two kernels
    b = pic.Run(pic.Params(npart=n, ncell=ng, length=L, block_size=256, **kw), device="cuda:0")
    x, v = state(n, 7 * n + ng)
    a.init(x, v)
    b.init(x, v)
    return a, b


def assert_same(a, b, n, ng):
    for p, q in zip(a.get_cells(), b.get_cells()):
        assert np.array_equal(p, q)
    f, g = a.get_field(), b.get_field()
    for k in ("rho_q", "E", "rho", "phi"):
        assert np.array_equal(f[k], g[k]), k
    d, e = a.diagnostics(), b.diagnostics()
    for k in ("step", "charge_q", "charge", "field"):
        assert np.array_equal(d[k], e[k]), k
    assert np.isnan(d["kinetic"][-1]) and np.isnan(d["momentum"][-1])
    # the kinetic sums and the modes add float32 terms in another order
    np.testing.assert_allclose(d["kinetic"][:-1], e["kinetic"][:-1], rtol=1e-5)
    scale = L / n * np.abs(a.get_cells()[1]).sum()
    assert np.abs(d["momentum"][:-1] - e["momentum"][:-1]).max(initial=0.0) <= 1e-5 * scale
    tol = 2.0 / ng * np.abs(f["E"]).sum() * 64 * 2.0 ** -24 + 1e-12
    assert np.abs(d["mode"][-1] - e["mode"][-1]).max() <= tol


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 1023, 1024, 1025, 131072, 131073, 700001])
@pytest.mark.parametrize("ng", [1, 2, 31, 32, 33, 256, 257, 512, 513, 1025, 4096])
def test_steps_equal_the_two_kernels(n, ng):
    a, b = pair(n, ng)
    for k in (1, 6, 2, 9):             # more steps than accumulators, and fewer
        a.step_n(k)
        b.step_n(k)
    assert_same(a, b, n, ng)


@pytest.mark.parametrize("n,ng,S", [(20000, 64, 1), (50021, 100, 3), (300007, 777, 7), (1000003, 2048, 20)])
@pytest.mark.parametrize("shape", [pic.PIC_SHAPE_CIC, pic.PIC_SHAPE_NGP])
def test_sorted_steps_equal_the_two_kernels(n, ng, S, shape):
    a, b = pair(n, ng, sort_interval=S, shape=shape)
    for k in (5, 1, 20, 3):
        a.step_n(k)
        b.step_n(k)
    assert_same(a, b, n, ng)
    a.push(), a.solve_field(), b.push(), b.solve_field()      # single phases in between
    a.step_n(4), b.step_n(4)
    assert_same(a, b, n, ng)


@pytest.mark.parametrize("n,ng", [(12500000, 2049), (12500001, 2049), (24000000, 512), (24000001, 512),
                                  (100003, 4096), (100003, 4097)])
def test_steps_at_the_limits_of_the_launch(n, ng):
    a, b = pair(n, ng)
    a.step_n(3), b.step_n(3)
    assert_same(a, b, n, ng)


def test_crowded_cells_and_a_steep_field():
    # all particles in one cell, and a plasma whose field spans its largest range
    n, ng = 262147, 1000
    for kw in (dict(), dict(rho_ion=1e-30), dict(rho_ion=1e25)):   # E32 near its smallest and largest
        a, b = pair(n, ng, **kw)
        x = np.full(n, 0.3, np.float32)
        for r in (a, b):
            r.set_state(x, np.zeros(n, np.float32), 5)
            r.step_n(3)
        for p, q in zip(a.get_cells(), b.get_cells()):
            assert np.array_equal(p, q, equal_nan=True)
        assert np.array_equal(a.get_field()["E"], b.get_field()["E"], equal_nan=True)


@pytest.mark.parametrize("bad", [float("nan"), float("-inf")])
def test_a_bad_particle_is_flagged_and_the_run_restarts(bad):
    a, b = pair(5001, 64)
    x, v = state(5001, 1)
    w = v.copy()
    w[5000] = bad
    a.set_state(x, w, 0)
    a.step_n(3)
    with pytest.raises(pic.PicError) as e:
        a.sync()
    assert e.value.code == pic.PIC_EDEVICE
    for r in (a, b):
        r.set_state(x, v, 0)
        r.step_n(7)
    assert_same(a, b, 5001, 64)


def test_a_captured_step_replays():
    a, b = pair(20000, 64)
    s = torch.cuda.Stream()
    c = pic.Run(pic.Params(npart=20000, ncell=64, length=L), device="cuda:0", stream=s)
    c.init(*state(20000, 7 * 20000 + 64))
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        c.step_n(1)
    for _ in range(4):
        g.replay()
    torch.cuda.synchronize()
    b.step_n(4)
    for p, q in zip(c.get_cells(), b.get_cells()):
        assert np.array_equal(p, q)


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 255, 257, 20000, 100003])
@pytest.mark.parametrize("ng", [1, 2, 31, 33, 64, 256, 257, 1000, 1024])
def test_float64_steps_equal_the_two_kernels(n, ng):
    # the float64 density is exact integers, so the launches agree bit for bit
    rng = np.random.default_rng(3 * n + ng)
    x = rng.uniform(0.0, L, n)
    x[:1] = 0.0
    x[1:2] = np.nextafter(L, 0.0)
    v = rng.normal(0.0, 0.4, n)
    runs = []
    for kw in (dict(), dict(block_size=256)):
        r = pic.Run(pic.Params(npart=n, ncell=ng, length=L, precision=pic.PIC_FP64, sort_interval=7, **kw),
                    device="cuda:0")
        r.init(x, v)
        for k in (1, 6, 2, 9):
            r.step_n(k)
        runs.append(r)
    a, b = runs
    for p, q in zip(a.get_state(), b.get_state()):
        assert np.array_equal(p, q)
    f, g = a.get_field(), b.get_field()
    for k in ("E", "rho", "phi"):
        assert np.array_equal(f[k], g[k]), k
    d, e = a.diagnostics(), b.diagnostics()
    for k in ("step", "charge", "field"):
        assert np.array_equal(d[k], e[k]), k
    np.testing.assert_allclose(d["kinetic"][:-1], e["kinetic"][:-1], rtol=1e-13)
    scale = L / n * np.abs(a.get_state()[1]).sum()
    assert np.abs(d["momentum"][:-1] - e["momentum"][:-1]).max() <= 1e-13 * scale
    assert np.isnan(d["kinetic"][-1])


@pytest.mark.parametrize("n,ng", [(1000000, 1024), (1000001, 1024), (65537, 256), (1000, 1025)])
def test_float64_steps_at_the_limits_of_the_launch(n, ng):
    rng = np.random.default_rng(n)
    x, v = rng.uniform(0.0, L, n), rng.normal(0.0, 0.2, n)
    out = []
    for kw in (dict(), dict(block_size=512)):
        r = pic.Run(pic.Params(npart=n, ncell=ng, length=L, precision=pic.PIC_FP64, **kw), device="cuda:0")
        r.init(x, v)
        r.step_n(3)
        out.append((*r.get_state(), r.get_field()["E"]))
    for p, q in zip(*out):
        assert np.array_equal(p, q)


@pytest.mark.parametrize("n,ng", [(40000, 256), (40001, 256), (40000, 257), (400000, 512), (400001, 512),
                                  (400001, 513), (600000, 1024), (600001, 1024), (600000, 1025)])
@pytest.mark.parametrize("shape", [pic.PIC_SHAPE_CIC, pic.PIC_SHAPE_NGP])
def test_steps_at_the_limits_of_one_particle_per_lane(n, ng, shape):
    # where the lanes' groups and the block size change; integers, so bit for bit
    a, b = pair(n, ng, shape=shape)
    for k in (1, 7):
        a.step_n(k), b.step_n(k)
        assert_same(a, b, n, ng)
    a.close(), b.close()


@pytest.mark.parametrize("n,ng", [(1, 1), (255, 1023), (20000, 64), (300007, 1024), (300007, 1025),
                                  (1000003, 2049), (70000, 8192)])
def test_a_sort_is_the_stable_order_by_cell(n, ng):
    # the passes run into each other: several sorts and pushes back to back
    run = pic.Run(pic.Params(npart=n, ncell=ng, length=L, sort_interval=8), device="cuda:0")
    run.init(*state(n, 3 * n + ng))
    u, v = run.get_cells()
    for _ in range(3):
        run.sort()
        order = np.argsort(np.clip(u, 0, ng - 1).astype(np.int64), kind="stable")
        u, v = u[order], v[order]
        got = run.get_cells()
        assert np.array_equal(got[0], u) and np.array_equal(got[1], v)
        run.push(), run.sort(), run.solve_field()
        w = run.get_cells()
        key = np.clip(w[0], 0, ng - 1).astype(np.int64)
        assert np.all(np.diff(key) >= 0)
        run.push(), run.solve_field()
        u, v = run.get_cells()
    run.close()


@pytest.mark.parametrize("n,ng", [(8388608, 4096), (8388609, 64), (8389631, 777), (9000001, 8192)])
@pytest.mark.parametrize("precision", [pic.PIC_FP32_FIXED, pic.PIC_FP64])
def test_a_sort_of_long_chunks_is_the_stable_order_by_cell(n, ng, precision):
    run = pic.Run(pic.Params(npart=n, ncell=ng, length=L, precision=precision, sort_interval=8), device="cuda:0")
    rng = np.random.default_rng(n)
    x = np.minimum(rng.uniform(0.0, L, n).astype(run.p.dtype), np.nextafter(run.p.dtype(L), run.p.dtype(0)))
    run.init(x, np.arange(n, dtype=run.p.dtype) * run.p.dtype(1e-9))
    if precision == pic.PIC_FP64:
        u, key = x, np.minimum((x * (ng / L)).astype(np.int64), ng - 1)
        take = lambda: run.get_state()[0]
    else:
        u = run.get_cells()[0]
        key = np.clip(u, 0, ng - 1).astype(np.int64)
        take = lambda: run.get_cells()[0]
    run.sort()
    assert np.array_equal(take(), u[np.argsort(key, kind="stable")])
    run.close()


@pytest.mark.parametrize("H", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("n,ng,precision", [(20000, 64, pic.PIC_FP32_FIXED), (300007, 777, pic.PIC_FP32_FIXED),
                                            (5001, 1025, pic.PIC_FP32_FIXED), (20000, 64, pic.PIC_FP64)])
def test_short_history_rings_hold_the_last_rows(H, n, ng, precision):
    # rows that share a slot of the ring are written in the steps' order
    rng = np.random.default_rng(H)
    dt = np.float64 if precision == pic.PIC_FP64 else np.float32
    x, v = rng.uniform(0.0, 0.999 * L, n).astype(dt), rng.normal(0.0, 0.4, n).astype(dt)
    runs = []
    for kw in (dict(), dict(block_size=256)):
        r = pic.Run(pic.Params(npart=n, ncell=ng, length=L, precision=precision, history=H, **kw), device="cuda:0")
        r.init(x, v)
        runs.append(r)
    for k in (1, 2, 5, 6, 7, 40):
        rows = []
        for r in runs:
            r.step_n(k)
            rows.append(r.diagnostics(max(0, r.step - H + 1), min(H, r.step + 1)))
        d, e = rows
        for key in ("step", "charge_q", "charge", "field"):
            assert np.array_equal(d[key], e[key]), key
        for key in ("kinetic", "momentum"):
            assert np.isnan(d[key][-1]) and np.all(np.isfinite(d[key][:-1]))
        np.testing.assert_allclose(d["kinetic"][:-1], e["kinetic"][:-1], rtol=1e-5)
        np.testing.assert_allclose(d["mode"], e["mode"], rtol=0, atol=64 * 2.0 ** -24 * 2.0 / ng *
                                   np.abs(runs[0].get_field()["E"]).sum() + 1e-12)
    for r in runs:
        r.close()


@pytest.mark.parametrize("H", [1, 2, 3])
def test_short_history_rings_of_a_pool(H):
    n, ng = 20000, 64
    p = pic.Params(npart=n, ncell=ng, length=L, history=H)
    x, v = state(n, 5)
    pool = pic.Pool(max_slots=1, ncell_max=ng, arena_bytes=1 << 24, history=H, device="cuda:0")
    slot = pool.admit(p, x, v, 30)
    run = pic.Run(pic.Params(npart=n, ncell=ng, length=L, history=H, block_size=256), device="cuda:0")
    run.init(x, v)
    for k in (1, 2, 7, 20):
        pool.advance(k)
        run.step_n(k)
        first, count = max(0, run.step - H + 1), min(H, run.step + 1)
        d, e = pool.diagnostics(slot, first, count), run.diagnostics(first, count)
        for key in ("step", "charge_q"):
            assert np.array_equal(d[key], e[key]), key
        np.testing.assert_allclose(d["field"], e["field"], rtol=1e-12)
        assert np.isnan(d["kinetic"][-1]) and np.all(np.isfinite(d["kinetic"][:-1]))
    pool.close()


@pytest.mark.parametrize("n", [1, 20, 45])
@pytest.mark.parametrize("kw", [{}, dict(sort_interval=3), dict(precision=pic.PIC_FP64), dict(block_size=128),
                                dict(block_size=128, sort_interval=20)])
def test_captured_steps_replay_and_the_run_goes_on(n, kw):
    # many steps in a capture, of runs that replay graphs of their own, too
    dt = np.float64 if kw.get("precision") == pic.PIC_FP64 else np.float32
    rng = np.random.default_rng(n)
    x, v = rng.uniform(0.0, 0.999 * L, 20000).astype(dt), rng.normal(0.0, 0.4, 20000).astype(dt)
    s = torch.cuda.Stream()
    a = pic.Run(pic.Params(npart=20000, ncell=64, length=L, **kw), device="cuda:0", stream=s)
    b = pic.Run(pic.Params(npart=20000, ncell=64, length=L, **{**kw, "block_size": 256}), device="cuda:0")
    a.init(x, v), b.init(x, v)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        a.step_n(n)
    # a sort swaps the buffers that the graph was captured with
    replays = 1 if "sort_interval" in kw else 3
    for _ in range(replays):
        g.replay()
    torch.cuda.synchronize()
    b.step_n(n * replays)
    a.step_n(7), b.step_n(7)
    for p, q in zip(a.get_state(), b.get_state()):
        assert np.array_equal(p, q)
    # the host counted the captured steps once; the device's rows are those of b
    rows = a.diagnostics(0, a.step + 1)
    want = b.diagnostics(0, a.step + 1)
    assert a.step == n + 7
    for key in ("step", "charge_q", "charge", "field"):
        assert np.array_equal(rows[key], want[key]), key
    a.close(), b.close()


@pytest.mark.parametrize("steps", [1, 2, 3, 20])
@pytest.mark.parametrize("H", [4, 64])
@pytest.mark.parametrize("phases", [False, True])
def test_steps_after_replays_continue_the_devices_count(steps, H, phases):
    # a short and a long ring; the device's step counter, read through the rows
    s = torch.cuda.Stream()
    a = pic.Run(pic.Params(npart=5001, ncell=64, length=L, history=H), device="cuda:0", stream=s)
    a.init(*state(5001, 9))
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        if phases:
            a.push(), a.solve_field()
        else:
            a.step_n(1)
    a.set_state(*state(5001, 9), 0)           # the graph is still there
    a.step_n(1)
    with torch.cuda.stream(s):                # a replay goes to the current stream
        for _ in range(H + 1):
            g.replay()
    a.step_n(steps)
    torch.cuda.synchronize()
    first = max(0, a.step - H + 1)
    held = a.diagnostics(first, a.step - first + 1)["step"]
    last = 1 + H + 1 + steps
    # the ring holds the device's last H rows
    slots = {r % H: r for r in range(max(0, last - H + 1), last + 1)}
    assert held.tolist() == [slots[r % H] for r in range(first, a.step + 1)]
    a.close()


@pytest.mark.parametrize("n,ng", [(300000, 512), (300001, 512), (600002, 1024), (600003, 1025), (600005, 100), (2, 1026),
                                  (3, 2049), (6, 4096)])
@pytest.mark.parametrize("shape", [pic.PIC_SHAPE_CIC, pic.PIC_SHAPE_NGP])
def test_the_last_particles_of_a_run_and_another_block_size(n, ng, shape):
    # 1 to 3 particles beyond the last group of 4, no group at all, and the lines of
    # steps_shape
    a, b = pair(n, ng, shape=shape, sort_interval=5)
    for k in (1, 3, 8):
        a.step_n(k), b.step_n(k)
        assert_same(a, b, n, ng)
    a.close(), b.close()


# Rows against float64 sums of the same particles.  Products and group sums are
# rounded to 2^-24 of themselves, a thread's sum once a group, at random: an error of
# the total of 2^-24 / 2 sqrt(adds in a chain / threads) rms, taken 8 times; chains
# and threads of the push kernels' sums, which the launch's may not exceed.
@pytest.mark.parametrize("n,ng", [(20000, 64), (300007, 300), (1024003, 1024), (4200001, 2048), (12345679, 4096),
                                  (23000003, 2000)])
@pytest.mark.parametrize("shape", [pic.PIC_SHAPE_CIC, pic.PIC_SHAPE_NGP])
def test_kinetic_energy_and_momentum_against_float64_sums(n, ng, shape):
    run = pic.Run(pic.Params(npart=n, ncell=ng, length=L, shape=shape), device="cuda:0")
    run.init(*state(n, 11))
    m = L / n
    threads = min(n / 4.0, 1536.0 * 152)
    tol = 8 * 2.0 ** -25 * math.sqrt(max(4.0, n / threads) / threads)
    old = run.get_cells()[1].astype(np.float64)
    for _ in range(4):
        run.step_n(1)
        new = run.get_cells()[1].astype(np.float64)
        row = run.diagnostics(run.step - 1, 1)[0]
        assert abs(row["kinetic"] - 0.5 * m * (old * new).sum()) <= tol * 0.5 * m * np.abs(old * new).sum()
        assert abs(row["momentum"] - m * new.sum()) <= tol * m * np.abs(new).sum()
        old = new
    run.close()


# Mode amplitudes against float64 sums: P = NG/256 parts are summed in float32, 13 adds
# deep, each rounding at random to 2^-25 of the part (rms 2^-25 / sqrt 3), at most
# 1/P of sum |E|; the parts' errors add in squares.
@pytest.mark.parametrize("n,ng", [(1000003, 2048), (4000001, 4096)])
def test_mode_amplitudes_against_float64_sums(n, ng):
    run = pic.Run(pic.Params(npart=n, ncell=ng, length=L), device="cuda:0")
    run.init(*state(n, 12))
    theta = 2.0 * math.pi * np.arange(ng) / ng
    parts, err = ng / 256.0, []
    for _ in range(12):
        run.step_n(1)
        E = run.get_field()["E"]
        row = run.diagnostics(run.step, 1)[0]
        for m in range(8):
            want = 2.0 / ng * abs(np.sum(E * np.exp(-1j * (m + 1) * theta)))
            err.append((row["mode"][m] - want) / (2.0 / ng * np.abs(E).sum()))
    assert np.sqrt(np.mean(np.square(err))) <= math.sqrt(13.0 / parts) * 2.0 ** -25 / math.sqrt(3.0)
    run.close()


def many_step_launched(run):
    """Whether pic_step_n takes the many-step launch: its waits are made to run out
    (the run needs a new state afterwards)."""
    run.set_wait_limit(4096, 1)
    run.step_n(2)
    try:
        run.sync()
        return False
    except pic.PicError as e:
        assert e.code == pic.PIC_ETIMEOUT
        return True
    finally:
        run.set_wait_limit()


@pytest.mark.parametrize("shape", [pic.PIC_SHAPE_CIC, pic.PIC_SHAPE_NGP])
@pytest.mark.parametrize("open_shape", [True, False])
def test_a_shape_from_the_tuning_cache_leaves_the_run_as_tuning_does(tmp_path, shape, open_shape):
    n, ng, path = 200003, 1024, str(tmp_path / "shapes.json")
    kw = dict() if open_shape else dict(block_size=128)
    runs = [pic.Run(pic.Params(npart=n, ncell=ng, length=L, shape=shape, **kw), device="cuda:0") for _ in range(2)]
    for i, r in enumerate(runs):
        r.init(*state(n, 4))
        assert (len(r.autotune(reps=2, cache=path)) == 0) == (i == 1)
        r.step_n(5)
    assert runs[0].launch_shape() == runs[1].launch_shape()
    assert_same(runs[0], runs[1], n, ng)
    assert [many_step_launched(r) for r in runs] == [open_shape, open_shape]
    r = pic.Run(pic.Params(npart=n, ncell=ng, length=L, shape=shape), device="cuda:0")
    r.init(*state(n, 4))
    r.set_launch(block=256)
    assert not many_step_launched(r)
    for bad in ((0, 256, 1), (3, 256, 1), (1, 0, 1), (1, 256, 3), (9, 512, 4)):
        assert pic._lib.pic_adopt_launch(r._h, *bad) == pic.PIC_EINVAL


@pytest.mark.parametrize("n,ng,shape,H", [(20000, 64, pic.PIC_SHAPE_CIC, 256), (300007, 777, pic.PIC_SHAPE_NGP, 256),
                                          (700001, 4096, pic.PIC_SHAPE_CIC, 3), (5, 1, pic.PIC_SHAPE_CIC, 1)])
def test_the_sort_interval_is_tuned_on_the_launch_that_the_run_takes(n, ng, shape, H):
    a, b = pair(n, ng, shape=shape, history=H)
    for r in (a, b):
        r.step_n(9)
    intervals = (0, 1, 20, 5)
    best, ms = a.tune_sort_interval(intervals)
    assert list(ms) == list(intervals) and all(t > 0 for t in ms.values())
    assert ms[best] == min(ms.values())
    # the state, the rows and the launch's own accumulators and counters are as before
    for _ in range(2):
        a.step_n(7), b.step_n(7)
        for p, q in zip(a.get_cells(), b.get_cells()):
            assert np.array_equal(p, q)
        f, g = a.get_field(), b.get_field()
        for k in ("rho_q", "E", "rho", "phi"):
            assert np.array_equal(f[k], g[k]), k
        first, count = max(0, a.step - H + 1), min(H, a.step + 1)
        d, e = a.diagnostics(first, count), b.diagnostics(first, count)
        for k in ("step", "charge_q", "field"):
            assert np.array_equal(d[k], e[k]), k
    a.phase_space(8, 8, -1.0, 1.0)
    a.tune_sort_interval((0, 10), adopt=True)
    a.step_n(25)
    a.sync()
    # timed in the launch that pic_step_n takes: its waits run out there too, and a
    # run whose shape is chosen has none
    for r, takes in ((a, True), (b, False)):
        r.set_wait_limit(4096, 1)
        if takes:
            with pytest.raises(pic.PicError) as e:
                r.tune_sort_interval(intervals)
            assert e.value.code == pic.PIC_ETIMEOUT
        else:
            r.tune_sort_interval(intervals)
    a.close(), b.close()


@pytest.mark.parametrize("threads", [False, True])
def test_runs_on_streams_of_their_own_equal_the_two_kernels(threads):
    # many-step launches of several runs in flight at once, one by one and from threads
    specs = [(20000, 64, 0), (300007, 500, 7), (1000003, 1024, 0), (700001, 4096, 0), (50021, 100, 3), (20000, 100, 0),
             (3, 1, 0), (131073, 2048, 5)]
    runs = []
    for i, (n, ng, S) in enumerate(specs):
        kw = dict(precision=pic.PIC_FP64) if i == 5 else {}
        r = pic.Run(pic.Params(npart=n, ncell=ng, length=L, sort_interval=S, **kw), device="cuda:0",
                    stream=torch.cuda.Stream())
        x, v = state(n, i)
        r.init(x.astype(r.p.dtype), v.astype(r.p.dtype))
        runs.append(r)

    def go(r):
        for k in (1, 30, 2, 17):
            r.step_n(k)
        r.sync()

    if threads:
        import threading
        ts = [threading.Thread(target=go, args=(r,)) for r in runs]
        [t.start() for t in ts], [t.join() for t in ts]
    else:
        for k in (1, 30, 2, 17):
            for r in runs:
                r.step_n(k)
    for i, (r, (n, ng, S)) in enumerate(zip(runs, specs)):
        q = pic.Run(pic.Params(npart=n, ncell=ng, length=L, sort_interval=S, precision=r.p.precision, block_size=256),
                    device="cuda:0")
        x, v = state(n, i)
        q.init(x.astype(q.p.dtype), v.astype(q.p.dtype))
        q.step_n(50)
        for a, b in zip(r.get_state(), q.get_state()):
            assert np.array_equal(a, b)
        assert np.array_equal(r.get_field()["E"], q.get_field()["E"])
        r.close(), q.close()


def test_handles_close_while_another_stream_is_captured():
    # more handles with page-locked slabs than are kept: the rest are freed
    runs = []
    for i in range(12):
        r = pic.Run(pic.Params(npart=1000, ncell=16, length=L), device="cuda:0")
        r.init(*state(1000, i))
        for _ in range(40):
            r.sync()
        runs.append(r)
    x = torch.zeros(16, device="cuda")
    s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):                  # "global" capture mode
        x.add_(1.0)
        for r in runs:
            pic._lib.pic_destroy(r._h)
            r._h = None
        x.add_(1.0)
    g.replay()
    torch.cuda.synchronize()
    assert torch.all(x == 2.0)
    r = pic.Run(pic.Params(npart=1000, ncell=16, length=L), device="cuda:0")
    r.init(*state(1000, 0))
    for _ in range(40):
        r.sync()
    assert len(r.diagnostics()) == 1
    r.close()


def test_a_call_beside_another_streams_capture_does_not_count_as_captured():
    # a run on the legacy stream cannot step while another stream is captured in the
    # default mode; afterwards it is as it was
    a, b = pair(20000, 64)
    s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    x = torch.zeros(4, device="cuda")
    torch.cuda.synchronize()
    failed = None
    try:
        with torch.cuda.graph(g, stream=s):
            x.add_(1.0)
            try:
                a.step_n(2)
            except pic.PicError as e:
                failed = e.code
    except RuntimeError:
        pass                                           # the capture is lost
    torch.cuda.synchronize()
    if failed is None:                                 # (where it can, it has stepped)
        b.step_n(2)
    a.step_n(3), b.step_n(3)
    assert_same(a, b, 20000, 64)
    assert many_step_launched(a)
