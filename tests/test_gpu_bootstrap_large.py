"""The signed bootstrap of a run large enough for the bucket-counting draws.

From 4e6 particles on, residual draws that fall into a guide-table bucket
inside one cell are counted by bucket in shared memory instead of added to
their cell one by one: the same integers as the oracle's, cell by cell.
"""
import os

import numpy as np
import pytest

import workloads
from helpers import make_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nk", [(100, 64), (3, 2), (700, 300)])
def test_large_bootstrap_matches_the_oracle(nx, nk):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_02121_gb300 import Simulation, build
    build.build()
    wl = workloads.scaled(workloads.GAUSS_2D_FP64_2E5, strategy="sp2", n_alpha=4_000_001, nx=nx,
                          nk=nk, xmin=-25.0, xmax=25.0, kmin=-3.2, kmax=3.2, resample_every=2)
    sim = Simulation(wl, 16_000_000)
    o = make_oracle(wl, threads=min(16, os.cpu_count() or 1))
    o.init_gauss(wl["n_alpha"], wl["x0"], wl["sigma_x"], wl["k0"])
    sim.run(2)
    o.step(2)
    o.annihilate()
    assert np.array_equal(sim.grid_counts(), o.grid())
    c = sim.counters()
    assert c["boot_nrplus"] > 0 and c["boot_nrminus"] > 0
    sim.close()
