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
