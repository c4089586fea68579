"""Batches whose replicas are large or crowded, against the oracle, bit for bit:
binary64 with two lanes and with one thread per cell, and shifts whose cells are
read before and after the draw is known."""
import numpy as np
import pytest

import oracle as O
from paper_1211_1646_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PREC = {"fp64": O.FP64, "fp32": O.FP32}


@pytest.mark.parametrize("prec,cells,shapes,nsel", [
    ("fp64", "sigma", [(541, 540), (94, 110)], 4),       # one thread per cell; shifts read late
    ("fp64", "sigma", [(541, 540), (94, 110)], 8),
    ("fp64", "sigma", [(541, 540), (37, 44)], 11),       # run-time n_M
    ("fp64", "sigma", [(300, 290), (40, 38)], 8),        # two lanes; shifts read early
    ("fp64", "sigma", [(301, 310), (203, 200), (5, 62)], 4),   # one thread; shifts read early
    ("fp64", "sqrt2", [(401, 420), (61, 62)], 5),        # crowded cells
    ("fp32", "sqrt2", [(401, 420), (61, 62)], 4),
    ("fp32", "sigma", [(541, 540), (94, 110)], 8),
])
def test_large_and_crowded_replicas(prec, cells, shapes, nsel):
    from paper_1211_1646_gb300 import build, hdmc
    build.build()
    reps = []
    for k, (nx, ny) in enumerate(shapes):
        Lx, Ly = W.hex_box(nx, ny, 0.723 if nx == 5 else 0.70)   # five columns: wide cells with up to four disks
        reps.append(W.Workload("r%d" % k, nx * ny, Lx, Ly, 0.11, nsel, 31 + k, 0))
    b = hdmc.Batch(reps, precision=prec, cells=cells)
    b.sweep(5)
    b.sample()
    hist = b.pressure()[2]
    for k, w in enumerate(reps):
        r = O.System(w.N, w.Lx, w.Ly, 1.0, w.d, nsel, w.seed, PREC[prec],
                     cells=O.CELLS_SQRT2 if cells == "sqrt2" else O.CELLS_SIGMA)
        r.sweep(5)
        loc, cnt = b.state(k)
        assert np.array_equal(cnt, r.state()[1])
        assert np.array_equal(loc, r.state()[0])
        assert np.array_equal(b.counters()[k], r.counters())
        assert np.array_equal(b.origin(k), r.origin())
        assert np.array_equal(hist[k], r.histogram())
