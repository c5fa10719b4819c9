"""The regeneration plan at the edges of its tiles.

A restored histogram's particles have to lie, slot after slot, in the cells
their counts give (Alg. 3 in cell order), with the counts' signs, in their
instances: for sizes around the plan's sub-tiles and its one-block limit, for
counts around a 32-slot tile and around the cells whose tiles are filled
apart, and for contexts of few and of many slots.
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


def histogram(kind, cells, rng):
    g = np.zeros(cells, np.int64)
    if kind == "ones":
        g[:] = 1
    elif kind == "edges":       # around one tile and around the dense cells' eight
        vals = [31, -32, 33, -255, 256, 257, 223, -224, 225, 1, 0, 0, -1, 5000]
        at = np.sort(rng.choice(cells, min(cells, 400), replace=False))
        g[at] = [vals[i % len(vals)] for i in range(len(at))]
    elif kind == "one cell":
        g[cells // 2] = -70_001
    elif kind == "ends":
        g[0], g[-1] = 3, -40
    elif kind == "mixed":
        g[:] = rng.integers(-2, 3, cells)
        g[rng.integers(0, cells, 5)] = 3000
    return g.astype(np.int32)


def check(x, k, s, g, wl):
    want = np.repeat(np.arange(g.size), np.abs(g))
    assert len(x) == len(want)
    ix = np.floor((x - wl["xmin"]) * (wl["nx"] / (wl["xmax"] - wl["xmin"]))).astype(int)
    ik = np.floor((k - wl["kmin"]) * (wl["nk"] / (wl["kmax"] - wl["kmin"]))).astype(int)
    assert np.array_equal(ix * wl["nk"] + ik, want % (wl["nx"] * wl["nk"]))
    assert np.array_equal(s, np.sign(g)[want])
    return want // (wl["nx"] * wl["nk"])


@pytest.mark.parametrize("kind", ["ones", "edges", "one cell", "ends", "mixed"])
@pytest.mark.parametrize("nx,nk", [(1, 1), (1, 31), (33, 62), (32, 64), (1, 2049), (128, 128),
                                   (5, 3277), (300, 101)])
def test_slots_lie_in_their_cells(nx, nk, kind):
    from paper_1709_02121_gb300 import Simulation
    g = histogram(kind, nx * nk, np.random.default_rng(nx * 1000 + nk))
    total = int(np.abs(g).sum())
    for capacity in (max(total, 64), 3_000_000):   # few tiles, and more than 65536
        wl = workloads.scaled(workloads.GAUSS_2D_FP64_2E5, n_alpha=10, nx=nx, nk=nk)
        sim = Simulation(wl, capacity)
        sim.restore(g.reshape(nx, nk), 10, 1)
        x, k, s, _, pid = sim.particles()
        check(x, k, s, g, wl)
        assert np.array_equal(pid, (1 << 40) + np.arange(total).astype(np.uint64))
        assert sim.counters()["nonzero_cells"] == np.count_nonzero(g)
        sim.close()


@pytest.mark.parametrize("ninst,nx,nk", [(256, 7, 1), (3, 20, 30), (70, 61, 57)])
def test_instances_own_their_slots(ninst, nx, nk):
    from paper_1709_02121_gb300 import Batch
    rng = np.random.default_rng(ninst)
    g = histogram("mixed", ninst * nx * nk, rng).reshape(ninst, nx * nk)
    g[rng.integers(0, ninst, ninst // 3)] = 0      # empty instances
    wl = workloads.scaled(workloads.GAUSS_2D_FP64_2E5, nx=nx, nk=nk)
    insts = [dict(H=1.0, w=1.0, x0=0.0, sigma_x=1.0, k0=1.0, n_init=0, n_alpha=1)] * ninst
    b = Batch(wl, insts, int(np.abs(g).sum()) + 100)
    b.restore(g.reshape(ninst, nx, nk), 10, 1)
    x, k, s, _, pid, inst = b.particles()
    want = check(x, k, s, g.reshape(-1), wl)
    assert np.array_equal(inst, want)
    first = np.searchsorted(want, np.arange(ninst))
    ids = (1 << 40) + (want << 32) + np.arange(len(want)) - first[want]
    assert np.array_equal(pid, ids.astype(np.uint64))
    b.close()
