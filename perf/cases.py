"""Performance cases of the library: what a user's program has it do, over the
range of sizes, precisions and options of the configurations in `bench.py` and
`workloads/`.

A case is a dict of plain values.  `prepare` makes the initial particles on
the GPU from the seed and builds the run, pool or server that a program keeps;
`run` is one pass through the public entry points; `exact` states the same
pass in float64 with plain torch.  Four kinds of program:

  steps     a `Run` advanced by `step_n(steps)`; the program then reads the
            history rows of those steps and the field, and holds the device's
            particle arrays (`read` false: the device arrays alone)
  whole     a run from start to end: upload of the particles from pinned host
            memory, `step_n`, history, a phase-space snapshot, and the final
            particles back into pinned memory
  ensemble  a `Pool` of independent runs advanced together, each run's history
            and particles read back
  served    a `Server` that takes a burst of requests to their end and keeps
            each one's particles and field
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1108_1954_gb300 as pic
from paper_1108_1954_gb300 import serve

TWO_PI = 2.0 * math.pi
BOX = 4.0 * math.pi            # the box of the two-stream runs
CORE_BOX = 3.1415              # the box per core of the weak-scaling workload
L2_BYTES = 126e6               # a state larger than this streams from memory in every step

PRECISION = {"fixed": pic.PIC_FP32_FIXED, "atomic": pic.PIC_FP32_ATOMIC, "fp64": pic.PIC_FP64}


def _steps(name, npart, ncell, steps, *, precision="fixed", solver="exact", shape="cic",
           length=BOX, v0=0.2, vth=0.01, modes=1, eps=1e-3, sort=0, read=True):
    c = dict(kind="steps", npart=npart, ncell=ncell, steps=steps, precision=precision,
             solver=solver, shape=shape, length=length, v0=v0, vth=vth, modes=modes, eps=eps,
             sort=sort, read=read)
    return dict(c, name=name) if name else c


def _whole(name, npart, ncell, steps, *, sort=20, bins=128):
    c = dict(kind="whole", npart=npart, ncell=ncell, steps=steps, precision="fixed",
             solver="exact", shape="cic", length=BOX, v0=0.2, vth=0.01, modes=8, eps=1e-4,
             sort=sort, bins=bins)
    return dict(c, name=name) if name else c


def _ensemble(name, runs, steps, *, ncell_max=2048, npart_max=1000000, draw_seed=0):
    c = dict(kind="ensemble", runs=runs, steps=steps, ncell_max=ncell_max, npart_max=npart_max,
             draw_seed=draw_seed)
    return dict(c, name=name) if name else c


def _served(name, requests, *, steps_max=200, ncell_max=4096, npart_max=4000000, draw_seed=0):
    c = dict(kind="served", requests=requests, steps_max=steps_max, ncell_max=ncell_max,
             npart_max=npart_max, draw_seed=draw_seed)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: the 20,000-electron run stepped one step at a time, as
        # a program does that acts between steps; launches and latency are all of it
        _steps("one_step", 20000, 64, 1, read=False),
        # a small run of odd size, 200 steps and their history: graphs of short kernels
        _steps("small_run", 50021, 100, 200),
        # the plain two-stream run in its own float64 precision, to its end
        _steps("small_run_fp64", 20000, 64, 200, precision="fp64"),
        # 16 cores' share of the weak-scaling workload: Maxwellian plasma, sorted
        # every 20 steps, the particles resident in L2
        _steps("weak_exact", 1024000, 1024, 100, length=16 * CORE_BOX, v0=0.0, vth=0.2, modes=0,
               sort=20),
        # the same with the paper's field solver, 150 CG iterations per step
        _steps("weak_cg", 1024000, 1024, 20, length=16 * CORE_BOX, v0=0.0, vth=0.2, modes=0,
               sort=20, solver="cg"),
        # a middling run of odd size with the nearest-grid-point shape
        _steps("ngp_run", 3000017, 777, 50, shape="ngp", sort=10),
        # the single large run: 2^26 electrons, modes 1..8, one sort period a pass
        _steps("large_run", 1 << 26, 4096, 20, modes=8, eps=1e-4, sort=20),
        # a whole program from pinned host memory and back, of odd size
        _whole("whole_program", 12345679, 4096, 20),
        # the precision study's float64 arm
        _steps("study_fp64", 1 << 24, 1024, 20, precision="fp64", vth=0.02, sort=20),
        # the precision study's float32-atomic arm, watched step by step
        _steps("study_atomic", 1 << 24, 1024, 1, precision="atomic", vth=0.02, sort=20,
               read=False),
        # the parameter sweep: 512 uneven runs in one pool, histories and particles read
        _ensemble("ensemble", 512, 100),
        # a burst of ten requests through the serving loop
        _served("served", 10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["one", "small", "small64", "weak", "cg", "ngp", "large", "whole", "fp64",
                       "atomic", "ensemble", "served"])
    vth = rng.uniform(0.005, 0.05)
    v0 = rng.uniform(0.05, 0.5)
    if kind == "one":
        return _steps(None, _log_int(rng, 1e4, 1e6), _log_int(rng, 64, 2048), 1, v0=v0, vth=vth,
                      read=False)
    if kind == "small":
        return _steps(None, _log_int(rng, 1e4, 5e5), _log_int(rng, 64, 2048),
                      rng.randint(50, 200), v0=v0, vth=vth, sort=rng.choice([0, 0, 10, 20]))
    if kind == "small64":
        return _steps(None, _log_int(rng, 1e4, 1e5), _log_int(rng, 64, 512), rng.randint(50, 200),
                      precision="fp64", v0=v0, vth=vth)
    if kind in ("weak", "cg"):
        p = _log_int(rng, 4, 128)
        return _steps(None, 64000 * p, 64 * p, rng.randint(20, 60) if kind == "weak" else
                      rng.randint(10, 20), length=CORE_BOX * p, v0=0.0, vth=0.2, modes=0, sort=20,
                      solver="exact" if kind == "weak" else "cg")
    if kind == "ngp":
        return _steps(None, _log_int(rng, 1e5, 2e7), _log_int(rng, 64, 8192), rng.randint(10, 40),
                      shape="ngp", v0=v0, vth=vth, sort=rng.choice([0, 10, 20]))
    if kind == "large":
        return _steps(None, _log_int(rng, 1e6, 6e7), _log_int(rng, 256, 8192), 20, v0=v0, vth=vth,
                      modes=8, eps=1e-4, sort=rng.choice([0, 10, 20, 40]))
    if kind == "whole":
        return _whole(None, _log_int(rng, 1e5, 3e7), _log_int(rng, 64, 8192), rng.randint(5, 40),
                      sort=rng.choice([0, 20]), bins=rng.choice([32, 64, 128]))
    if kind == "fp64":
        return _steps(None, _log_int(rng, 1e5, 1.6e7), _log_int(rng, 64, 4096), 20,
                      precision="fp64", v0=v0, vth=vth, sort=rng.choice([0, 20]))
    if kind == "atomic":
        return _steps(None, _log_int(rng, 1e6, 1.6e7), _log_int(rng, 256, 4096), 1,
                      precision="atomic", v0=v0, vth=vth, sort=20, read=False)
    if kind == "ensemble":
        return _ensemble(None, _log_int(rng, 8, 400), rng.randint(20, 100),
                         draw_seed=rng.randint(1, 10 ** 6))
    return _served(None, rng.randint(2, 10), draw_seed=rng.randint(1, 10 ** 6))


# --- inputs -------------------------------------------------------------------

def _generator(seed, *more):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(np.random.default_rng([int(seed), *more]).integers(1 << 62)))
    return g


def _particles(npart, length, v0, vth, nmodes, eps, gen):
    """Float64 (x, v) on the GPU: a lattice displaced by modes 1..nmodes of
    density amplitude eps with random phases, beams +-v0 by particle parity
    with thermal spread vth."""
    j = torch.arange(npart, device="cuda", dtype=torch.float64)
    x0 = (j + 0.5) * (length / npart)
    x = x0.clone()
    phases = (TWO_PI * torch.rand(max(nmodes, 1), generator=gen, device="cuda",
                                  dtype=torch.float64)).tolist()
    for m in range(1, nmodes + 1):
        k = TWO_PI * m / length
        x -= (eps / k) * torch.sin(k * x0 + phases[m - 1])
    x = torch.remainder(x, length)
    v = vth * torch.randn(npart, generator=gen, device="cuda", dtype=torch.float64)
    v += v0 * (1.0 - 2.0 * torch.remainder(j, 2.0))
    return x, v


def _state(npart, length, v0, vth, nmodes, eps, gen, double):
    """The particles as the program hands them over: CPU tensors in the run's
    precision, every position in [0, L)."""
    x, v = _particles(npart, length, v0, vth, nmodes, eps, gen)
    if not double:
        x, v = x.float(), v.float()
    x = torch.where((x >= 0) & (x < (length if double else float(np.float32(length)))), x,
                    torch.zeros_like(x))
    return x, v


def _host(t):
    out = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    out.copy_(t)
    return out


def _params(c, steps):
    return pic.Params(npart=c["npart"], ncell=c["ncell"], length=c["length"], dt=0.1,
                      precision=PRECISION[c["precision"]], sort_interval=c["sort"],
                      history=max(256, 2 * steps),
                      field_solver=pic.PIC_SOLVER_CG if c["solver"] == "cg"
                      else pic.PIC_SOLVER_EXACT,
                      shape=pic.PIC_SHAPE_NGP if c["shape"] == "ngp" else pic.PIC_SHAPE_CIC)


def _run_state(c, seed):
    return _state(c["npart"], c["length"], c["v0"], c["vth"], c["modes"], c["eps"],
                  _generator(seed, 1), c["precision"] == "fp64")


def _ensemble_runs(c):
    """The sweep's runs, from the case alone: cells and particles spread over
    their logarithm, beam and thermal speeds uniform (configuration ranges of
    `workloads.ensemble_runs`)."""
    r = np.random.default_rng([c["draw_seed"], 3])
    n = c["runs"]
    ncell = np.exp(r.uniform(math.log(64), math.log(c["ncell_max"]), n)).round().astype(int)
    npart = np.exp(r.uniform(math.log(1e4), math.log(c["npart_max"]), n)).round().astype(int)
    v0, vth = r.uniform(0.05, 0.5, n), r.uniform(0.001, 0.05, n)
    return [dict(npart=int(npart[i]), ncell=int(ncell[i]), length=BOX, v0=float(v0[i]),
                 vth=float(vth[i]), steps=c["steps"]) for i in range(n)]


def _served_requests(c, seed):
    """The burst's requests (ranges of `workloads.request_stream`, steps up to
    `steps_max`), with loading seeds from the seed."""
    r = np.random.default_rng([c["draw_seed"], 5])
    n = c["requests"]
    ncell = np.exp(r.uniform(math.log(64), math.log(c["ncell_max"]), n)).round().astype(int)
    npart = np.exp(r.uniform(math.log(1e4), math.log(c["npart_max"]), n)).round().astype(int)
    steps = r.integers(c["steps_max"] // 4, c["steps_max"] + 1, n)
    seeds = np.random.default_rng([int(seed), 7]).integers(1, 1 << 62, n)
    return [dict(npart=int(npart[i]), ncell=int(ncell[i]), length=BOX, v0=0.2, vth=0.01,
                 steps=int(steps[i]), seed=int(seeds[i])) for i in range(n)]


SERVED_MODES = ((1, 1e-3, 0.5),)


def prepare(case, seed):
    c = case
    if c["kind"] in ("steps", "whole"):
        x, v = _run_state(c, seed)
        run = pic.Run(_params(c, c["steps"]))
        s = dict(case=c, run=run)
        if c["kind"] == "whole":
            s.update(x0=_host(x), v0=_host(v), x=torch.empty_like(x, device="cpu", pin_memory=True),
                     v=torch.empty_like(v, device="cpu", pin_memory=True))
        else:
            run.init(x.cpu(), v.cpu())
            if not c["read"]:
                s["views"] = run.device_arrays()
        return s
    if c["kind"] == "ensemble":
        runs = _ensemble_runs(c)
        hist = max(128, c["steps"] + 1)
        ps = [pic.Params(npart=r["npart"], ncell=r["ncell"], length=r["length"], dt=0.1)
              for r in runs]
        nbytes = sum(pic.pool_run_bytes(p, hist) for p in ps) + (64 << 20)
        pool = pic.Pool(max_slots=len(ps), ncell_max=c["ncell_max"], arena_bytes=nbytes,
                        history=hist)
        slots = []
        for i, (p, r) in enumerate(zip(ps, runs)):
            x, v = _state(r["npart"], r["length"], r["v0"], r["vth"], 1, 1e-3,
                          _generator(seed, 2, i), False)
            slots.append(pool.admit(p, x.cpu(), v.cpu(), 1 << 40))
        pool.advance(0)
        total = sum(r["npart"] for r in runs)
        x = torch.empty(total, dtype=torch.float32, pin_memory=True)
        v = torch.empty(total, dtype=torch.float32, pin_memory=True)
        sizes = [r["npart"] for r in runs]
        return dict(case=c, pool=pool, slots=slots, x=x, v=v, xs=x.split(sizes), vs=v.split(sizes))
    reqs = _served_requests(c, seed)
    requests = [serve.Request(i, 0.0, pic.Params(npart=r["npart"], ncell=r["ncell"],
                                                 length=r["length"], dt=0.1),
                              pic.Loading(v0=r["v0"], vth=r["vth"], seed=r["seed"],
                                          modes=SERVED_MODES), r["steps"])
                for i, r in enumerate(reqs)]
    nbytes = sum(pic.pool_run_bytes(r.params, 8) for r in requests) + (64 << 20)
    server = serve.Server(arena_bytes=nbytes, max_slots=64, ncell_max=c["ncell_max"])
    return dict(case=c, server=server, requests=requests)


# --- one pass -----------------------------------------------------------------

def _rows(rows, double):
    """The history as a program keeps it.  The float32 modes sum the kinetic
    energy in float32 per thread, and every mode the mode amplitudes from
    float32 terms, so those are kept as float32.  The momentum is left out: the
    two beams' sums cancel, and what remains has no accuracy relative to
    itself."""
    f = np.float64 if double else np.float32
    return dict(kinetic=rows["kinetic"].astype(f), field=rows["field"].copy(),
                mode=rows["mode"].astype(np.float32))


def run(state):
    s, c = state, state["case"]
    if c["kind"] == "steps":
        r = s["run"]
        if not c["read"]:
            r.step_n(c["steps"])
            x, v, e = s["views"] if c["sort"] == 0 else r.device_arrays()
            return dict(x=x, v=v, E=e)
        first = r.step
        r.step_n(c["steps"])
        rows = r.diagnostics(first, c["steps"])
        f = r.get_field()
        x, v, _ = r.device_arrays()
        out = dict(x=x, v=v, E=f["E"], phi=f["phi"], rho=f["rho"],
                   **_rows(rows, c["precision"] == "fp64"))
        if c["precision"] == "fixed":
            out.update(rho_q=f["rho_q"], charge_q=rows["charge_q"].copy())
        return out
    if c["kind"] == "whole":
        r = s["run"]
        r.init(s["x0"], s["v0"])
        r.step_n(c["steps"])
        rows = r.diagnostics(0, c["steps"])
        counts = r.phase_space(c["bins"], c["bins"], -0.6, 0.6)
        x, v = r.get_state(s["x"], s["v"])
        return dict(x=x, v=v, counts=counts.astype(np.int64), charge_q=rows["charge_q"].copy(),
                    **_rows(rows, False))
    if c["kind"] == "ensemble":
        pool = s["pool"]
        first = pool.step_count(s["slots"][0])
        pool.advance(c["steps"])
        rows = []
        for slot, x, v in zip(s["slots"], s["xs"], s["vs"]):
            rows.append(pool.diagnostics(slot, first, c["steps"]))
            pool.get_state(slot, x, v)
        rows = np.concatenate(rows)
        return dict(x=s["x"], v=s["v"], charge_q=rows["charge_q"].copy(), **_rows(rows, False))
    records, _ = s["server"].serve(s["requests"], keep=[r.rid for r in s["requests"]])
    out = []
    for rec in records:
        (x, v), f, _ = rec.result
        out.append(dict(x=x, v=v, E=f["E"], phi=f["phi"], rho=f["rho"], rho_q=f["rho_q"]))
    return out


# --- what a pass cannot do without ----------------------------------------------

def _work_one(npart, ncell, steps, wide, iterations=0):
    es = 8 if wide else 4
    once = 2.0 * npart * 2 * es                    # x, v read and written
    times = steps if npart * 2 * es > L2_BYTES else 1
    # gather 4, kick 2, drift 2, wrap 2, deposit 5, energies 3 a particle; the field
    # about 20 a node and 9 a node and iteration of the CG
    flops = steps * (18.0 * npart + (20.0 + 9.0 * iterations) * ncell)
    return dict(bytes=once * times + steps * 8.0 * ncell, flops=flops)


def work(case):
    c = case
    if c["kind"] in ("steps", "whole"):
        w = _work_one(c["npart"], c["ncell"], c["steps"], c["precision"] == "fp64",
                      150 if c["solver"] == "cg" else 0)
        if c["kind"] == "whole":                   # up, down, and the snapshot's read
            w["bytes"] += 24.0 * c["npart"]
        return w
    runs = _ensemble_runs(c) if c["kind"] == "ensemble" else _served_requests(c, 0)
    parts = [_work_one(r["npart"], r["ncell"], r["steps"], False) for r in runs]
    state = 8.0 * sum(r["npart"] for r in runs)
    if c["kind"] == "ensemble" and state > L2_BYTES:   # all runs advance together
        parts = [dict(bytes=16.0 * r["npart"] * r["steps"], flops=p["flops"])
                 for r, p in zip(runs, parts)]
    return dict(bytes=sum(p["bytes"] for p in parts) + state, flops=sum(p["flops"] for p in parts))


# --- the same in float64, by plain torch -----------------------------------------

def _deposit(x, ncell, length, shape):
    s = x * (ncell / length)
    if shape == "ngp":
        return torch.bincount(torch.remainder(s.floor().long(), ncell), minlength=ncell).double()
    s = s - 0.5
    fl = s.floor()
    f = s - fl
    left = torch.remainder(fl.long(), ncell)
    w = torch.bincount(left, weights=1.0 - f, minlength=ncell)
    return w + torch.bincount(torch.remainder(left + 1, ncell), weights=f, minlength=ncell)


def _cg(rho, dx, iterations):
    """The paper's conjugate gradient with Phi_0 = 0 pinned, from Phi = 0."""
    n = rho.numel()
    r = -rho * dx * dx
    r[0] = 0.0
    x, v, c = torch.zeros_like(r), r.clone(), r @ r
    for _ in range(iterations):
        z = -2.0 * v
        z[1:] += v[:-1]
        z[:-1] += v[1:]
        z[0] = v[0]
        if n > 1:
            z[-1] = v[-2] - 2.0 * v[-1]
        t = c / (z @ v)
        x += t * v
        r = r - t * z
        d = r @ r
        v = (d / c) * v + r
        c = d
    return x


def _field(x, c):
    n, ng, dx = x.numel(), c["ncell"], c["length"] / c["ncell"]
    rho = 1.0 - _deposit(x, ng, c["length"], c.get("shape", "cic")) * (ng / n)
    if c.get("solver") == "cg":
        phi = _cg(rho, dx, 150)
        e = -(torch.roll(phi, -1) - torch.roll(phi, 1)) / (2.0 * dx)
        return rho, phi, e
    s = torch.cumsum(rho, 0)
    s = s - s.mean()
    e = 0.5 * dx * (s + torch.roll(s, 1))
    phi = -dx * dx * (torch.cumsum(s, 0) - s)
    return rho, phi, e


def _gather(x, e, c):
    s = x * (c["ncell"] / c["length"])
    if c.get("shape") == "ngp":
        return e[torch.remainder(s.floor().long(), c["ncell"])]
    s = s - 0.5
    fl = s.floor()
    left = torch.remainder(fl.long(), c["ncell"])
    el = e[left]
    return el + (s - fl) * (e[torch.remainder(left + 1, c["ncell"])] - el)


def _simulate(x, v, c):
    """`steps` steps from float64 (x, v) in physical units, with their history rows."""
    length, ng, n = c["length"], c["ncell"], x.numel()
    dx, mass = length / ng, length / n
    theta = (TWO_PI / ng) * torch.arange(ng, device=x.device, dtype=torch.float64)
    waves = torch.stack([torch.exp(-1j * m * theta) for m in range(1, 9)])
    rows = dict(kinetic=[], field=[], mode=[])
    rho, phi, e = _field(x, c)
    for _ in range(c["steps"]):
        vn = v - 0.1 * _gather(x, e, c)
        rows["kinetic"].append(0.5 * mass * (v * vn).sum())
        rows["field"].append(0.5 * dx * (e * e).sum())
        rows["mode"].append((waves @ e.to(torch.complex128)).abs() * (2.0 / ng))
        v = vn
        x = torch.remainder(x + 0.1 * v, length)
        x = torch.where(x >= length, torch.zeros_like(x), x)
        rho, phi, e = _field(x, c)
    return x, v, rho, phi, e, {k: torch.stack(t) for k, t in rows.items()}


def _splitmix64(seed, k):
    def shr(z, b):
        return (z >> b) & ((1 << (64 - b)) - 1)

    def wrap(a):
        return a - (1 << 64) if a >= 1 << 63 else a
    z = wrap(seed & ((1 << 64) - 1)) + k * wrap(0x9E3779B97F4A7C15)
    z = (z ^ shr(z, 30)) * wrap(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * wrap(0x94D049BB133111EB)
    return shr(z ^ shr(z, 31), 40).double()


def _loaded(r):
    """The loader's two-stream state (include/pic.h, pic_loading) in float64,
    rounded to float32 as the loader hands it over."""
    n, length = r["npart"], r["length"]
    j = torch.arange(n, device="cuda", dtype=torch.int64)
    x0 = (j.double() + 0.5) * (length / n)
    x = x0.clone()
    for m, eps, phase in SERVED_MODES:
        k = TWO_PI * m / length
        x -= (eps / k) * torch.sin(k * x0 + phase)
    u1 = (_splitmix64(r["seed"], 2 * j + 1) + 1.0) * 2.0 ** -24
    u2 = _splitmix64(r["seed"], 2 * j + 2) * 2.0 ** -24
    g = torch.sqrt(-2.0 * torch.log(u1)) * torch.cos(TWO_PI * u2)
    v = r["vth"] * g + r["v0"] * (1.0 - 2.0 * (j % 2).double())
    return torch.remainder(x, length).float().double(), v.float().double()


def exact(case, seed):
    c = case
    if c["kind"] in ("steps", "whole"):
        x, v = _run_state(c, seed)
        x, v, rho, phi, e, rows = _simulate(x.double(), v.double(), c)
        if 0 < c["sort"] < c["steps"]:
            # sorted on the way: one particle whose rounded position lies in another
            # cell moves all the others in the arrays
            x = v = None
        if c["kind"] == "whole":
            return dict(x=x, v=v, counts=None, charge_q=None, **rows)
        if c["precision"] != "fp64" and x is not None:   # the device keeps cell coordinates
            x = x * (c["ncell"] / c["length"])
        if not c["read"]:
            return dict(x=x, v=v, E=e)
        out = dict(x=x, v=v, E=e, phi=phi, rho=rho, **rows)
        return dict(out, rho_q=None, charge_q=None) if c["precision"] == "fixed" else out
    if c["kind"] == "ensemble":
        runs = _ensemble_runs(c)
        if len(runs) * c["steps"] > 6400:          # half a million kernels and more: over 20 s
            return None
        xs, vs, rows = [], [], []
        for i, r in enumerate(runs):
            x, v = _state(r["npart"], r["length"], r["v0"], r["vth"], 1, 1e-3,
                          _generator(seed, 2, i), False)
            x, v, _, _, _, h = _simulate(x.double(), v.double(), r)
            xs.append(x)
            vs.append(v)
            rows.append(h)
        return dict(x=torch.cat(xs), v=torch.cat(vs), charge_q=None,
                    **{k: torch.cat([h[k] for h in rows]) for k in rows[0]})
    out = []
    for r in _served_requests(c, seed):
        x, v = _loaded(r)
        x, v, rho, phi, e, _ = _simulate(x, v, r)
        out.append(dict(x=x, v=v, E=e, phi=phi, rho=rho, rho_q=None))
    return out
