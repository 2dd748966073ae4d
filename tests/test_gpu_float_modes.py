"""The float64 and float32-atomic pushes at the sizes where their groups, tiles
and integer locate can go wrong, against the FP64 oracle.

float64: the deposit is exact integers of 2^-53, so the density is compared with
exactly summed weights (the oracle's own sums are rounded at every add): what
is left is the result's rounding, n/ng 2^-52 a node at most, and the cell
fraction's ng 2^-52 per particle.  float32 atomic: a node's float32
sum is off by at most its number of adds times its size times 2^-24, and the
fraction by ng 2^-24."""
import math

import numpy as np
import pytest

import oracle as O
import paper_1108_1954_gb300 as pic
import torch  # noqa: F401

pytestmark = pytest.mark.gpu
L = 3.7


def state(n, ng, seed):
    """Random particles, with some on nodes, cell edges and the box's ends."""
    rng = np.random.default_rng(seed)
    x = rng.uniform(0.0, L, n)
    dx = L / ng
    edge = [0.0, np.nextafter(0.0, 1.0), np.nextafter(L, 0.0), 0.5 * dx, np.nextafter(0.5 * dx, 0.0),
            L - 0.5 * dx, (ng // 2) * dx]
    k = min(n, len(edge))
    x[:k] = edge[:k]
    return np.clip(x, 0.0, np.nextafter(L, 0.0)), rng.normal(0.0, 0.3, n)


def exact_density(x, ng):
    """rho from the CIC weights of x, summed without rounding: the weights as
    multiples of 2^-52, their halves of 26 bits summed exactly in float64."""
    s = x * (ng / L) - 0.5
    left = np.floor(s).astype(np.int64)
    w = np.rint((s - left) * 2.0 ** 52).astype(np.int64)
    total = np.zeros(ng)
    for node, q in ((left % ng, (1 << 52) - w), ((left + 1) % ng, w)):
        total += np.bincount(node, (q >> 26).astype(float), ng) * 2.0 ** -26 \
            + np.bincount(node, (q & ((1 << 26) - 1)).astype(float), ng) * 2.0 ** -52
    return 1.0 - total * (ng / x.size)


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 7, 255, 256, 257, 2051, 40003])
@pytest.mark.parametrize("ng", [1, 2, 3, 64, 127, 128, 1000, 8191, 8192])
def test_fp64_step_at_the_edges(n, ng):
    x, v = state(n, ng, 31 * n + ng)
    run = pic.Run(pic.Params(npart=n, ncell=ng, length=L, precision=pic.PIC_FP64), device="cuda:0")
    run.init(x, v)
    ref = O.State(O.params(ng, n, L, 0.1), x, v)
    tol = (n / ng + ng * math.sqrt(n) + 8) * 2.0 ** -50 * (ng / n)
    assert np.abs(run.get_field()["rho"] - exact_density(x, ng)).max() <= tol
    assert abs(run.get_field()["rho"].sum()) <= 1e-12          # every particle whole
    run.push()
    run.solve_field()
    ref.step()
    x1, v1 = run.get_state()
    d = np.abs(x1 - ref.x)
    assert np.minimum(d, L - d).max() <= 1e-12 * L
    assert np.abs(v1 - ref.v).max() <= 1e-11
    assert abs(run.get_field()["rho"].sum()) <= 1e-12


@pytest.mark.parametrize("n", [1, 3, 4, 5, 257, 40003])
@pytest.mark.parametrize("ng", [1, 64, 574, 575, 1150, 8192])     # 32, 16, 8 and 2 copies
def test_atomic_deposit_at_the_edges(n, ng):
    x, v = state(n, ng, 17 * n + ng)
    x32 = np.minimum(x.astype(np.float32), np.nextafter(np.float32(L), np.float32(0)))
    run = pic.Run(pic.Params(npart=n, ncell=ng, length=L, precision=pic.PIC_FP32_ATOMIC),
                  device="cuda:0")
    run.init(x32, v.astype(np.float32))
    ref = O.State(O.params(ng, n, L, 0.1), x32.astype(np.float64), v)
    most = float((1.0 - ref.rho).max() / (ng / n))              # the fullest node's particles
    tol = (ng / n) * 2.0 ** -24 * (2.0 * (most + 1) ** 2 + 2.0 * ng * (most + 1))
    assert np.abs(run.get_field()["rho"] - ref.rho).max() <= tol
    run.push()
    run.solve_field()
    u1, _ = run.get_cells()
    assert ((u1 >= 0) & (u1 < ng)).all()


@pytest.mark.parametrize("precision", [pic.PIC_FP64, pic.PIC_FP32_ATOMIC])
@pytest.mark.parametrize("bad", [float("nan"), float("-inf"), -1e4])   # (beyond the far end is the point 0)
def test_a_particle_thrown_out_of_the_box_is_flagged(precision, bad):
    n = 1001
    x, v = state(n, 64, 5)
    v[n - 1] = v[500] = bad                                     # in a group and in the tail
    run = pic.Run(pic.Params(npart=n, ncell=64, length=L, precision=precision), device="cuda:0")
    dt = run.p.dtype
    run.init(np.minimum(x.astype(dt), np.nextafter(dt(L), dt(0))), v.astype(dt))
    run.push()
    with pytest.raises(pic.PicError) as e:
        run.sync()
    assert e.value.code == pic.PIC_EDEVICE


@pytest.mark.parametrize("n,ng", [(1, 1), (7, 2), (1000, 3), (100003, 100), (100003, 1024), (300001, 8192)])
def test_float64_sort_is_the_stable_order_by_cell(n, ng):
    # cell edges and their neighbours among the positions; the key is that of
    # plain float64 arithmetic, so the order is the same particle for particle
    rng = np.random.default_rng(n + ng)
    x, v = state(n, ng, n)
    k = n // 2
    edge = rng.integers(0, ng + 1, k) / (ng / L)
    x[n - k:] = np.clip(np.nextafter(edge, edge + rng.choice([-1.0, 0.0, 1.0], k)), 0.0, np.nextafter(L, 0.0))
    run = pic.Run(pic.Params(npart=n, ncell=ng, length=L, precision=pic.PIC_FP64, sort_interval=4),
                  device="cuda:0")
    run.init(x, v)
    run.sort()
    order = np.argsort(np.minimum((x * (ng / L)).astype(np.int64), ng - 1), kind="stable")
    assert np.array_equal(run.get_state()[0], x[order])
    run.close()


@pytest.mark.parametrize("n", [311295, 311300, 400003])       # below and at a block of 1024 for every SM
@pytest.mark.parametrize("ng", [574, 575, 1674, 1675, 8192])  # copies 32/32, 16/32, 8/32, 8/16, 2/4
def test_atomic_deposit_in_large_blocks(n, ng):
    # the density and the next step's against blocks of 512 threads: two orders of
    # the same float32 adds, each within the bound above of the exact sum
    x, v = state(n, ng, n + ng)
    x32 = np.minimum(x.astype(np.float32), np.nextafter(np.float32(L), np.float32(0)))
    rho = []
    for block in (0, 512):
        run = pic.Run(pic.Params(npart=n, ncell=ng, length=L, precision=pic.PIC_FP32_ATOMIC, block_size=block),
                      device="cuda:0")
        run.init(x32, v.astype(np.float32))
        rho.append([run.get_field()["rho"]])
        run.step_n(1)
        rho[-1].append(run.get_field()["rho"])
        run.close()
    for a, b in zip(*rho):
        most = float((1.0 - np.minimum(a, b)).max() / (ng / n))
        assert np.abs(a - b).max() <= 2 * (ng / n) * 2.0 ** -24 * (2.0 * (most + 1) ** 2 + 2.0 * ng * (most + 1))
        assert abs(a.sum()) <= 2 * ng * (ng / n) * 2.0 ** -24 * 2.0 * (most + 1) ** 2


# Rows of the float32-atomic mode against float64 sums of the same particles.  A
# float32 rounding of p is off by p 2^-24 / sqrt 3 rms at most; what is rounded is each
# product, and beyond 2^22 particles the sums of 2, 3 and 4 of a group: for particles
# of one size sqrt(1 + 4 + 9 + 16) / 2 times as much.  The rows' rms over 12 steps.
@pytest.mark.parametrize("n,ng", [(20001, 64), (1000003, 1024), (1 << 22, 512), ((1 << 22) + 1, 512), ((1 << 23) + 3, 1024)])
def test_atomic_rows_against_float64_sums(n, ng):
    rng = np.random.default_rng(n)
    run = pic.Run(pic.Params(npart=n, ncell=ng, length=L, precision=pic.PIC_FP32_ATOMIC), device="cuda:0")
    run.init(rng.uniform(0.0, 0.999 * L, n).astype(np.float32), rng.normal(0.3, 0.2, n).astype(np.float32))
    err = {"kinetic": [], "momentum": []}
    old = run.get_cells()[1].astype(np.float64)
    for _ in range(12):
        run.step_n(1)
        new = run.get_cells()[1].astype(np.float64)
        row = run.diagnostics(run.step - 1, 1)[0]
        for key, p, k in (("kinetic", old * new, 0.5 * L / n), ("momentum", new, L / n)):
            rounding = 2.0 ** -24 / math.sqrt(3.0) * math.sqrt((p * p).sum()) * (1.0 if n <= 1 << 22 else 30 ** 0.5 / 2)
            err[key].append((row[key] / k - p.sum()) / rounding)
        old = new
    assert np.sqrt(np.mean(np.square(err["kinetic"]))) <= 1.0
    assert np.sqrt(np.mean(np.square(err["momentum"]))) <= 1.0
    run.close()
