"""Flights that run as one launch give the launch-per-round schedule's results.

Every source (regeneration, the arrays) and sink (histogram, weight sums, the
arrays) of the models that have a one-launch kernel, bit for bit, for few
particles (part-filled passes, idle warps) and for more than one pass a warp;
and a rate at which the one-launch kernels of the general contexts step back.
"""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

KEYS = ("events", "kill_plus", "kill_minus", "out_plus", "out_minus", "particle_steps",
        "particle_steps_first", "live", "step", "epoch", "candidates", "first_pairs")

BASE = dict(nx=100, nk=64, xmin=-25.0, xmax=25.0, kmin=-3.2, kmax=3.2, resample_every=5)


@pytest.fixture(scope="module", autouse=True)
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_02121_gb300 import build
    build.build()
    torch.cuda.set_device(0)
    return torch


def pair(torch, make):
    a, b = make(torch.cuda.Stream()), make(torch.cuda.Stream())
    b.one_launch_periods(False)
    return a, b


def same_particles(a, b):
    pa, pb = a.particles(), b.particles()
    ia, ib = np.argsort(pa[4], kind="stable"), np.argsort(pb[4], kind="stable")
    for u, v in zip(pa, pb):
        assert np.array_equal(u[ia], v[ib])


@pytest.mark.parametrize("n", [1, 33, 5000, 300_000])
@pytest.mark.parametrize("precision,strategy,td", [
    ("fp64", "sp1", False), ("fp64", "wp", False), ("fp32", "sp1", True), ("fp32", "wp", True),
    ("fp32", "sp1", False)])
def test_periods_and_steps(torch, n, precision, strategy, td):
    from paper_1709_02121_gb300 import Simulation
    wl = workloads.scaled(workloads.GAUSS_2D_FP64_2E5, precision=precision, strategy=strategy,
                          n_alpha=n, **BASE)
    if td:
        wl["comps"] = (dict(a=0.7, b=0.3, om=1.0, ph=0.5, w=0.8, xc=-10.0),
                       dict(a=-0.4, b=0.0, om=0.0, ph=0.0, w=1.2, xc=2.0))
    a, b = pair(torch, lambda st: Simulation(wl, 8 * n + 400_000, stream=st))
    for s in (a, b):
        s.graph(True)
        s.run(5)              # from the arrays into the histogram
        s.run(10)             # regenerated
    assert np.array_equal(a.grid_counts(), b.grid_counts())
    ca, cb = a.counters(), b.counters()
    assert [ca[k] for k in KEYS] == [cb[k] for k in KEYS]
    for s in (a, b):
        s.step(3)             # from the arrays into the arrays
    same_particles(a, b)
    for s in (a, b):
        s.annihilate()
    assert np.array_equal(a.grid_counts(), b.grid_counts())
    ca, cb = a.counters(), b.counters()
    assert [ca[k] for k in KEYS] == [cb[k] for k in KEYS]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_batches(torch, precision):
    from paper_1709_02121_gb300 import Batch
    wl = workloads.scaled(workloads.GAUSS_2D_FP64_2E5, precision=precision, **BASE)
    insts = [dict(H=h, w=v, xc=0.0, x0=-5.0, sigma_x=1.0, k0=1.5, n_init=m, n_alpha=max(m, 1))
             for h, v, m in ((1.0, 1.0, 7000), (0.6, 1.4, 0), (-1.5, 0.8, 37), (1.2, 0.7, 900))]
    a, b = pair(torch, lambda st: Batch(wl, insts, 500_000, stream=st))
    for s in (a, b):
        s.run(15)
        s.step(2)
    same_particles(a, b)
    ca, cb = a.counters(), b.counters()
    assert [ca[k] for k in KEYS] == [cb[k] for k in KEYS]


def test_high_rates_run_launch_per_round(torch):
    """P(candidate) above 1/2 per interval: a general context's flights keep
    the launch-per-round schedule (with its recursive drain)."""
    from paper_1709_02121_gb300 import Simulation
    wl = workloads.scaled(workloads.GAUSS_2D_FP64_2E5, n_alpha=500, gamma0=9.0, **BASE)
    a, b = pair(torch, lambda st: Simulation(wl, 400_000, stream=st))
    for s in (a, b):
        s.step(2)
        s.annihilate()
    assert np.array_equal(a.grid_counts(), b.grid_counts())
    assert a.counters()["launches"] == b.counters()["launches"]


@pytest.mark.parametrize("n", [2000, 120_000])
def test_a_full_queue_is_reported(torch, n):
    """Growth beyond the capacity ends the flight with the capacity error in
    either schedule (the excess is dropped, the launch ends by itself)."""
    from paper_1709_02121_gb300 import Simulation, WbrwError, wbrw
    wl = workloads.scaled(workloads.GAUSS_2D_FP64_2E5, precision="fp32", n_alpha=n, **BASE)
    wl["resample_every"] = 0
    for one in (True, False):
        sim = Simulation(wl, n + 50)
        sim.one_launch_periods(one)
        with pytest.raises(WbrwError) as ei:
            sim.step(9)
            sim.density()
        assert ei.value.status == wbrw.ERR_CAPACITY
        sim.close()
