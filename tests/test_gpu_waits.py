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
