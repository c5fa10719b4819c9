"""Annihilation of particles in the arrays: the histogram is the particles'.

Grids up to the size that fits shared memory are binned there; the cell of
every particle and the tallies outside the grid are computed here from the
materialised particles with the same operations, so the counts are equal.
"""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_02121_gb300 import build
    build.build()
    torch.cuda.set_device(0)
    return torch


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n", [99_999, 100_000, 700_001])
@pytest.mark.parametrize("nx,nk", [(1, 1), (100, 64), (320, 160), (321, 160)])
def test_histogram_of_the_arrays(precision, n, nx, nk):
    from paper_1709_02121_gb300 import Simulation
    # a narrow window: particles outside it on every side
    wl = workloads.scaled(workloads.GAUSS_2D_FP64_2E5, precision=precision, n_alpha=n, nx=nx,
                          nk=nk, x0=-1.0, xmin=-3.0, xmax=2.5, kmin=1.3, kmax=1.8)
    sim = Simulation(wl, 4 * n + 100_000)
    sim.step(2)
    x, k, s, _, _ = sim.particles()
    sim.annihilate()
    f = np.float64 if precision == "fp64" else np.float32
    ix = np.floor((x - f(wl["xmin"])) * f(nx / (wl["xmax"] - wl["xmin"])))
    ik = np.floor((k - f(wl["kmin"])) * f(nk / (wl["kmax"] - wl["kmin"])))
    inside = (ix >= 0) & (ix < nx) & (ik >= 0) & (ik < nk)
    cell = (ix * nk + ik)[inside].astype(np.int64)
    want = np.bincount(cell, weights=s[inside].astype(float), minlength=nx * nk)
    assert np.array_equal(sim.grid_counts().reshape(-1), want.astype(np.int64))
    c = sim.counters()
    assert c["out_plus"] == int(np.sum(~inside & (s > 0)))
    assert c["out_minus"] == int(np.sum(~inside & (s < 0)))
    sim.close()
