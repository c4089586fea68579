"""Diameters far from 1: the same chain as the oracle's, bit for bit, in every
form of the sub-sweep.  The binary32 estimates that settle clear cases in
binary64 have errors that grow with sigma^2, so their bands must too; and the
sentinel of an unused slot must stay out of reach."""
import numpy as np
import pytest

import oracle as O
from paper_1211_1646_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PREC = {"fp64": O.FP64, "fp32": O.FP32}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1211_1646_gb300 import build
    build.build()


def _same(g, r):
    lg, cg = g.state()
    lr, cr = r.state()
    assert np.array_equal(cg, cr)
    assert np.array_equal(lg, lr)
    assert np.array_equal(g.counters(), r.counters())


@pytest.mark.parametrize("sigma", [1e-15, 1e-6, 0.05, 300.0, 3000.0])
@pytest.mark.parametrize("prec,nx,ny,phi,cells,nsel,sweeps", [
    ("fp64", 94, 110, 0.70, "sigma", 4, 60),      # 8 lanes per cell
    ("fp64", 61, 62, 0.72, "sqrt2", 4, 100),      # 8 lanes, crowded cells
    ("fp64", 233, 254, 0.70, "sigma", 4, 10),     # 4 lanes
    ("fp64", 331, 350, 0.70, "sigma", 4, 5),      # 2 lanes
    ("fp64", 401, 420, 0.716, "sqrt2", 4, 5),     # 2 lanes, crowded cells
    ("fp64", 531, 560, 0.70, "sigma", 4, 2),      # one thread, n_M fixed
    ("fp64", 541, 540, 0.70, "sigma", 8, 1),
    ("fp64", 551, 544, 0.60, "sigma", 11, 1),     # one thread, run-time n_M
    ("fp32", 94, 110, 0.70, "sigma", 4, 60),
    ("fp32", 61, 62, 0.72, "sqrt2", 4, 100),
])
def test_disks(prec, nx, ny, phi, cells, nsel, sweeps, sigma):
    from paper_1211_1646_gb300 import hdmc
    Lx, Ly = W.hex_box(nx, ny, phi)
    a = (nx * ny, Lx * sigma, Ly * sigma, sigma, 0.11 * sigma, nsel, 23)
    g = hdmc.System(*a, prec, cells=cells)
    r = O.System(*a, PREC[prec], cells=O.CELLS_SQRT2 if cells == "sqrt2" else O.CELLS_SIGMA)
    g.sweep(sweeps)
    r.sweep(sweeps)
    _same(g, r)
    g.sample()
    assert np.array_equal(g.pressure()[2], r.histogram(200, 1e-4))


@pytest.mark.parametrize("sigma", [0.05, 300.0])
def test_batch_of_binary64_replicas(sigma):
    from paper_1211_1646_gb300 import hdmc
    reps = []
    for k, (nx, ny, phi) in enumerate([(40, 38, 0.70), (94, 110, 0.68)]):
        Lx, Ly = W.hex_box(nx, ny, phi)
        reps.append(W.Workload("r%d" % k, nx * ny, Lx * sigma, Ly * sigma, 0.11 * sigma, 4, 7 + k, 0))
    b = hdmc.Batch(reps, sigma=sigma, precision="fp64")
    b.sweep(60)
    for k, w in enumerate(reps):
        r = O.System(w.N, w.Lx, w.Ly, sigma, w.d, 4, w.seed, O.FP64)
        r.sweep(60)
        assert np.array_equal(b.state(k)[0], r.state()[0])
        assert np.array_equal(b.counters()[k], r.counters())


@pytest.mark.parametrize("sigma", [1e-6, 0.05, 300.0, 3000.0])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("q,sweeps", [(8, 60), (22, 4), (34, 2)])   # 32, 8, and 4 or 2 lanes per cell
def test_spheres(prec, q, sweeps, sigma):
    from paper_1211_1646_gb300 import hdmc
    w = W.fcc3(q, 0.47, 0.1)
    L = [x * sigma for x in w.L]
    g = hdmc.System3(w.N, L, sigma, 0.1 * sigma, 4, 11, prec)
    r = O.System3(w.N, L, sigma, 0.1 * sigma, 4, 11, PREC[prec])
    g.sweep(sweeps)
    r.sweep(sweeps)
    _same(g, r)
    g.sample()
    assert np.array_equal(g.pressure()[2], r.histogram(200, 1e-4))
