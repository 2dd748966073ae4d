"""The waits between a kernel's blocks run out: the launch ends, the host sees
PIC_ETIMEOUT, and the run goes on from a new state.  (The waits expect one arrival
more than there are, and give up after 20 ms or so.)"""
import math
import time

import numpy as np
import pytest

import paper_1108_1954_gb300 as pic
import torch  # noqa: F401

pytestmark = pytest.mark.gpu
L = 4.0 * math.pi
POLLS = 20000


def state(n, seed, dt=np.float32):
    rng = np.random.default_rng(seed)
    return rng.uniform(0.0, 0.999 * L, n).astype(dt), rng.normal(0.0, 0.2, n).astype(dt)


# the many-step launches (groups of one and of four, 1 to 4 nodes a thread, one and
# two diagnostics blocks), and the CG with one warp a block, with sums taken by every
# warp and by one
@pytest.mark.parametrize("n,ng,kw", [
    (20000, 64, {}), (20000, 64, dict(history=4)), (700001, 1024, {}), (300007, 2048, {}), (300007, 4096, {}),
    (20000, 100, dict(precision=pic.PIC_FP64)), (3, 1, {}),
    (20000, 33, dict(field_solver=pic.PIC_SOLVER_CG)), (20000, 1024, dict(field_solver=pic.PIC_SOLVER_CG)),
    (20000, 8192, dict(field_solver=pic.PIC_SOLVER_CG)),
    (20000, 777, dict(field_solver=pic.PIC_SOLVER_CG, precision=pic.PIC_FP64))])
def test_a_wait_that_runs_out_is_reported_and_the_run_restarts(n, ng, kw):
    dt = np.float64 if kw.get("precision") == pic.PIC_FP64 else np.float32
    x, v = state(n, n + ng, dt)
    a, b = (pic.Run(pic.Params(npart=n, ncell=ng, length=L, **kw), device="cuda:0") for _ in range(2))
    a.init(x, v), b.init(x, v)
    a.step_n(3)
    a.sync()
    a.set_wait_limit(POLLS, 1)
    t0 = time.perf_counter()
    a.step_n(2)
    with pytest.raises(pic.PicError) as e:
        a.sync()
    assert e.value.code == pic.PIC_ETIMEOUT
    assert time.perf_counter() - t0 < 5.0
    a.set_wait_limit()
    with pytest.raises(pic.PicError):                # until the run gets a state
        a.get_state()
    a.set_state(x, v, 0)
    for k in (1, 7):
        a.step_n(k), b.step_n(k)
    for p, q in zip(a.get_state(), b.get_state()):
        assert np.array_equal(p, q)
    assert np.array_equal(a.get_field()["E"], b.get_field()["E"])
    a.close(), b.close()


def test_wait_limits_are_checked():
    r = pic.Run(pic.Params(npart=10, ncell=4, length=L), device="cuda:0")
    for bad in ((-1, 0), (1, 0), (4095, 0), (0, 2), (0, -1)):
        with pytest.raises(pic.PicError) as e:
            r.set_wait_limit(*bad)
        assert e.value.code == pic.PIC_EINVAL
    r.set_wait_limit(4096, 0)
    r.close()


def test_a_pool_loses_the_runs_of_a_launch_whose_wait_ran_out():
    ps = [pic.Params(npart=n, ncell=ng, length=L) for n, ng in ((20000, 64), (300007, 1025), (5001, 300))]
    pool = pic.Pool(max_slots=4, ncell_max=2048, arena_bytes=1 << 26, history=16, device="cuda:0")
    first = pool.admit(ps[2], *state(5001, 2), 4)          # done before the others come
    pool.advance(4)
    kept = pool.get_state(first)
    slots = [pool.admit(p, *state(p.npart, i), 9) for i, p in enumerate(ps[:2])]
    pool.advance(3)
    pool.set_wait_limit(POLLS, 1)
    with pytest.raises(pic.PicError) as e:
        pool.advance(6)
    assert e.value.code == pic.PIC_ETIMEOUT
    pool.set_wait_limit()
    assert pool.finished() == [first]
    for s in slots:
        assert pool.step_count(s) == 3
        for read in (pool.get_state, pool.get_cells, pool.get_field, lambda s: pool.diagnostics(s, 3, 1)):
            with pytest.raises(pic.PicError) as e:
                read(s)
            assert e.value.code == pic.PIC_ETIMEOUT
    pool.sync()                                            # the word is clear, the other run readable
    for a, b in zip(pool.get_state(first), kept):
        assert np.array_equal(a, b)
    assert pool.advance(6) == 0
    for s in slots:
        pool.release(s)
    again = pool.admit(ps[1], *state(300007, 1), 5)
    assert pool.advance(9) == 1 and sorted(pool.finished()) == sorted([first, again])
    run = pic.Run(ps[1], device="cuda:0")
    run.init(*state(300007, 1))
    run.step_n(5)
    for a, b in zip(pool.get_cells(again), run.get_cells()):
        assert np.array_equal(a, b)
    assert np.array_equal(pool.get_field(again)["E"], run.get_field()["E"])
