"""The work that users of this package have it do, as cases that can be timed.

A case is one pass of a running simulation: the caller holds a context with
its buffers and a checkpointed histogram, resumes from the checkpoint, runs
one or more resampling periods (or plain intervals and one resampling), and
reads the observables the run is for.  `transmission` is the exception: the
differentiable call makes its own context each time.

Every pass starts from the same checkpoint, so it can be repeated, and its
result depends on the seed alone (the random streams are keyed by particle
and interval).  The checkpoint is taken while the packet meets the barrier:
particles of both signs, with the spread of cells and signs of a real run.
"""
import functools
import math

import numpy as np
import torch

from paper_1709_02121_gb300 import Batch, Simulation, Simulation4
from paper_1709_02121_gb300.grad import transmission
from paper_1709_02121_gb300.wbrw import wbrw_density

# Shared by the 2D cases: hbar = m = 1, the phase-space window of the 2D
# workloads, gamma0 at its default (the majorant rate).
BASE = dict(hbar=1.0, mass=1.0, gamma0=0.0, xc=0.0, sigma_x=2.5,
            xmin=-60.0, xmax=60.0, kmin=-6.4, kmax=6.4)


def listed():
    return [
        # The smallest call in use: the short FP32 run of the smoke check
        # (interactive use and tests), eight periods, replayed from graphs.
        dict(name="sp1 fp32 2e4 short", kind="period", precision="fp32", strategy="sp1", n=20000,
             nx=96, nk=64, dt=0.1, every=5, periods=8, H=1.0, w=1.0, k0=1.5, x0=-6.0, warm=4,
             graph=True),
        # A parameter study's ordinary run on a grid of odd sizes.
        dict(name="sp1 fp32 1.2e6 odd", kind="period", precision="fp32", strategy="sp1",
             n=1234567, nx=601, nk=257, dt=0.05, every=10, periods=4, H=1.0, w=1.0, k0=1.5,
             x0=-6.0, warm=6, graph=True),
        # The 2D workload at scale: one period of 1e8 particles.
        dict(name="sp1 fp32 1e8", kind="period", precision="fp32", strategy="sp1", n=100000000,
             nx=1200, nk=512, dt=0.05, every=10, periods=1, H=1.0, w=1.0, k0=1.5, x0=-6.0,
             warm=6, graph=True),
        # The same barrier with the signed bootstrap between periods.
        dict(name="sp2 fp32 3e7", kind="period", precision="fp32", strategy="sp2", n=30000000,
             nx=1200, nk=512, dt=0.05, every=10, periods=1, H=1.0, w=1.0, k0=1.5, x0=-6.0,
             warm=6, graph=True),
        # Weighted particles, launched eagerly.
        dict(name="wp fp32 1e7", kind="period", precision="fp32", strategy="wp", n=10000000,
             nx=1200, nk=512, dt=0.05, every=10, periods=1, H=1.0, w=1.0, k0=1.5, x0=-6.0,
             warm=6, graph=False),
        # The FP64 run of the 2D workload (2e5 particles, 240 x 128 cells).
        dict(name="sp1 fp64 2e5", kind="period", precision="fp64", strategy="sp1", n=200000,
             nx=240, nk=128, dt=0.1, every=10, periods=3, H=1.0, w=1.0, k0=1.5, x0=-6.0, warm=6,
             graph=True),
        # The switched double barrier (time-dependent potential).
        dict(name="td fp32 1e7", kind="td", n=10000000, nx=1200, nk=512, dt=0.05, every=10,
             periods=1, k0=1.5, x0=-15.0, warm=6, graph=True),
        # Plain intervals of a short collision and one resampling: the
        # particles live in the arrays, as in a run without a period.
        dict(name="steps fp32 1e6", kind="steps", precision="fp32", strategy="sp1", n=1000000,
             nx=240, nk=128, dt=0.05, steps=10, H=1.0, w=1.0, k0=1.5, x0=-6.0),
        # Many uneven independent problems in the same launches (a quarter of
        # the particles of the batched workload).
        dict(name="batch sp1 256", kind="batch", strategy="sp1", instances=256, n_lo=2500.0,
             n_hi=1.0e6, nx=600, nk=256, dt=0.05, every=10, periods=1, warm=4),
        # The same with the signed bootstrap of each instance.
        dict(name="batch sp2 64", kind="batch", strategy="sp2", instances=64, n_lo=10000.0,
             n_hi=1.0e6, nx=600, nk=256, dt=0.05, every=10, periods=1, warm=4),
        # The 4D Helium-like system at scale.
        dict(name="he4d fp32 5e7", kind="he4d", n=50000000, nx=64, nk=64, ny=4096, nkap=2048,
             dt=0.02, every=10, periods=1, warm=3),
        # T(H, w) and its derivatives at a few parameter points, forward and
        # backward: the whole differentiable call, its context included.
        dict(name="grad fp32 4x1e6", kind="grad", points=4, n=1000000, nx=240, nk=128, dt=0.025,
             every=16, steps=64, x0=-3.0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _grid(rng, n):
    """Cells per axis for n particles: several particles per cell, or the
    annihilation would not hold the particle count."""
    cells = max(2000.0, min(700000.0, n / rng.uniform(4.0, 60.0)))
    nx = int(math.sqrt(cells * rng.uniform(1.5, 2.5)))
    return nx, max(31, int(cells / nx))


def draw(rng):
    """One more case of the ranges that the listed ones stand for."""
    kind = rng.choice(["period", "period", "period", "td", "steps", "batch", "he4d", "grad"])
    if kind == "period":
        strategy = rng.choice(["sp1", "sp1", "sp2", "wp"])
        precision = rng.choice(["fp32", "fp32", "fp64"])
        n = int(_log(rng, 1.5e4, 4.0e5 if precision == "fp64" else 3.0e7))
        nx, nk = _grid(rng, n)
        return dict(kind=kind, precision=precision, strategy=strategy, n=n, nx=nx, nk=nk,
                    dt=rng.uniform(0.03, 0.06), every=rng.randint(4, 11),
                    periods=rng.randint(1, 4) if n < 3.0e6 else 1, H=rng.uniform(0.5, 1.4),
                    w=rng.uniform(0.6, 2.0), k0=rng.uniform(1.0, 2.5), x0=-6.0,
                    warm=rng.randint(2, 6), graph=rng.random() < 0.6)
    if kind == "td":
        n = int(_log(rng, 3.0e4, 1.5e7))
        nx, nk = _grid(rng, n)
        return dict(kind=kind, n=n, nx=nx, nk=nk, dt=rng.uniform(0.03, 0.06),
                    every=rng.randint(4, 10), periods=1, k0=rng.uniform(1.0, 2.5), x0=-15.0,
                    warm=rng.randint(2, 6), graph=rng.random() < 0.6)
    if kind == "steps":
        precision = rng.choice(["fp32", "fp32", "fp64"])
        n = int(_log(rng, 2.0e4, 3.0e5 if precision == "fp64" else 1.0e7))
        nx, nk = _grid(rng, n)
        return dict(kind=kind, precision=precision, strategy=rng.choice(["sp1", "sp1", "sp2"]),
                    n=n, nx=nx, nk=nk, dt=rng.uniform(0.03, 0.06), steps=rng.randint(1, 11),
                    H=rng.uniform(0.5, 1.4), w=rng.uniform(0.6, 2.0), k0=rng.uniform(1.0, 2.5),
                    x0=-6.0)
    if kind == "batch":
        n_lo = _log(rng, 2.0e3, 2.0e4)
        return dict(kind=kind, strategy=rng.choice(["sp1", "sp1", "sp2", "wp"]),
                    instances=int(_log(rng, 2.0, 256.0)), n_lo=n_lo, n_hi=n_lo * _log(rng, 2.0, 50.0),
                    nx=rng.randint(101, 601), nk=rng.randint(63, 257), dt=0.05,
                    every=rng.randint(5, 10), periods=1, warm=rng.randint(2, 4))
    if kind == "he4d":
        g = rng.choice([16, 21, 32, 33, 48])
        return dict(kind=kind, n=int(_log(rng, max(2.0e5, 3.0 * g ** 4), 3.0e7)), nx=g,
                    nk=g + rng.randint(0, 5), ny=rng.choice([1024, 1500, 4096]),
                    nkap=rng.choice([512, 777, 2048]), dt=0.02, every=rng.randint(4, 10),
                    periods=1, warm=2)
    every = rng.randint(8, 16)  # (T is read right after a resampling)
    return dict(kind="grad", points=rng.randint(1, 9), n=int(_log(rng, 1.0e5, 1.0e6)),
                nx=rng.randint(100, 240), nk=rng.randint(64, 128), dt=0.025, every=every,
                steps=every * rng.randint(1, 4), x0=-3.0)


@functools.lru_cache(maxsize=None)
def _stream():
    """The program's own stream (graph replay needs a created one)."""
    return torch.cuda.Stream()


def _capacity(n):
    return int((4.0 if n <= 3.0e7 else 3.0) * n) + (1 << 20)


def _workload(case, seed, **more):
    wl = dict(BASE, precision=case.get("precision", "fp32"), strategy=case.get("strategy", "sp1"),
              dt=case["dt"], resample_every=case.get("every", 0), nx=case["nx"], nk=case["nk"],
              H=case.get("H", 1.0), w=case.get("w", 1.0), k0=case.get("k0", 1.5),
              x0=case.get("x0", -15.0), n_alpha=case.get("n", 1), seed=int(seed))
    wl.update(more)
    return wl


def _pinned(nx, nk):
    t = [torch.empty(m, dtype=torch.float64, pin_memory=True) for m in (nx * nk, nx)]
    return t, [v.numpy() for v in t]


def _resume_point(sim, cells):
    """The histogram of the last resampling in device memory, and its place in time."""
    grid = torch.empty(cells, dtype=torch.int32, device="cuda")
    torch.cuda.current_stream().synchronize()
    _, step, epoch = sim.checkpoint(grid)
    return grid, step, epoch


def _points(case, seed):
    """Parameter points (H, w) of the differentiable call."""
    rng = np.random.default_rng(seed)
    return rng.uniform(0.6, 1.4, case["points"]), rng.uniform(0.6, 1.6, case["points"])


def prepare(case, seed):
    kind = case["kind"]
    state = dict(case=case)
    if kind == "grad":
        H, w = (torch.tensor(v, dtype=torch.float64, requires_grad=True)
                for v in _points(case, seed))
        wl = _workload(case, seed, sigma_x=1.0, xmin=-20.0, xmax=20.0)
        total = case["points"] * case["n"]
        return dict(state, H=H, w=w, wl=wl, capacity=6 * total + (1 << 20))
    if kind == "batch":
        rng = np.random.default_rng(seed)
        m = case["instances"]
        H, w, k0 = rng.uniform(0.5, 1.5, m), rng.uniform(0.5, 2.0, m), rng.uniform(1.0, 2.5, m)
        n = np.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]), m)).astype(int)
        insts = [dict(H=float(a), w=float(b), xc=0.0, x0=-6.0, sigma_x=2.5, k0=float(c),
                      n_init=int(d), n_alpha=int(d)) for a, b, c, d in zip(H, w, k0, n)]
        wl = _workload(case, seed)
        cap = _capacity(int(n.sum())) + 8 * m * case["nx"] * case["nk"] // 4
        sim = Batch(wl, insts, capacity=cap, stream=_stream())
        sim.graph(True)
        cells = m * case["nx"] * case["nk"]
    elif kind == "he4d":
        wl = dict(dim=4, Z=2.0, a=1.0, lam=1.0, xc=0.0, ny=case["ny"], nkap=case["nkap"],
                  x0=(-1.0, 1.0), sigma_x=1.0, k0=(0.5, -0.5), n_alpha=case["n"], dt=case["dt"],
                  resample_every=case["every"], nx=case["nx"], nk=case["nk"], xmin=-10.0,
                  xmax=10.0, kmin=-6.4, kmax=6.4, precision="fp32", strategy="sp1",
                  seed=int(seed), hbar=1.0, mass=1.0, gamma0=0.0)
        sim = Simulation4(wl, capacity=_capacity(case["n"]), stream=_stream())
        sim.graph(True)
        cells = (case["nx"] * case["nk"]) ** 2
    else:
        wl = _workload(case, seed)
        if kind == "td":
            wl["comps"] = (dict(a=0.4, b=0.4, om=0.1, ph=math.pi, w=2.0, xc=-10.0),
                           dict(a=0.8, b=0.0, om=0.0, ph=0.0, w=2.0, xc=10.0))
        sim = Simulation(wl, capacity=_capacity(case["n"]), stream=_stream())
        if case.get("graph"):
            sim.graph(True)
        cells = case["nx"] * case["nk"]
    if kind == "steps":
        sim.step(4)
        sim.annihilate()
    else:
        sim.run(case["warm"] * case["every"])
    grid, step, epoch = _resume_point(sim, cells)
    keep, views = _pinned(case["nx"], case["nk"])
    return dict(state, sim=sim, grid=grid, step=step, epoch=epoch, keep=keep, views=views)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "grad":
        H, w = state["H"], state["w"]
        H.grad = w.grad = None
        T = transmission(H, w, state["wl"], case["steps"], state["capacity"])
        T.sum().backward()
        return dict(T=T.detach(), dH=H.grad, dw=w.grad)
    sim = state["sim"]
    sim.restore(state["grid"], state["step"], state["epoch"])
    if kind == "steps":
        sim.step(case["steps"])
        sim.annihilate()
    else:
        sim.run(case["periods"] * case["every"])
    if kind == "batch":
        return dict(grid=sim.grid, T=sim.transmissions())
    dens, marg, T, live = wbrw_density(sim.ctx, sim.nx, sim.nk, *state["views"])
    return dict(grid=sim.grid, density=dens, marginal=marg, T=T, live=live)


def _size(case):
    """(particles, histogram cells, intervals, histograms made) of one pass."""
    kind = case["kind"]
    if kind == "grad":
        return (case["points"] * case["n"], case["points"] * case["nx"] * case["nk"], case["steps"],
                max(1, case["steps"] // case["every"]))
    if kind == "batch":
        r = math.log(case["n_hi"] / case["n_lo"])
        mean = (case["n_hi"] - case["n_lo"]) / r if r > 0 else case["n_lo"]
        return (int(case["instances"] * mean), case["instances"] * case["nx"] * case["nk"],
                case["every"] * case["periods"], case["periods"])
    cells = (case["nx"] * case["nk"]) ** (2 if kind == "he4d" else 1)
    if kind == "steps":
        return case["n"], cells, case["steps"], 1
    return case["n"], cells, case["every"] * case["periods"], case["periods"]


def work(case):
    """The histogram read and written and the observables written once; per
    particle and period one counter-based draw (ten rounds of two multiplies
    and four logical operations, the high and low words counted apart: 80
    operations) and its flight (about 20), and per expected candidate event
    1.6 draws and about 60 operations for the kick and the offspring."""
    n, cells, steps, made = _size(case)
    rate = {"td": 1.6, "he4d": 4.0}.get(case["kind"], case.get("H", 1.0))
    events = n * rate * case["dt"] * steps
    return dict(bytes=8.0 * cells + 8.0 * case["nx"] * case["nk"],
                flops=100.0 * n * made + 190.0 * events)


def exact(case, seed):
    """Monte Carlo counts: there is no value in closed form to hold them to."""
    return None
