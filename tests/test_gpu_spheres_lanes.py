"""The sphere sub-sweep in each of its lane groups (32, 8 and 4 or 2 lanes per
cell, chosen by the number of active cells) against the oracle, bit for bit:
state, slot order, counters."""
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


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("q,phi,nsel,sweeps", [
    (8, 0.42, 1, 6),      # 32 lanes per cell, wide cells (216 active cells)
    (8, 0.45, 20, 3),     # more trials than directions drawn ahead
    (20, 0.47, 4, 4),     # the last size of 32 lanes per cell (4096 active cells)
    (21, 0.47, 7, 3),     # 8 lanes per cell, 4913 active cells: a last block of one cell
    (30, 0.45, 9, 2),     # 8 lanes per cell, chunked directions, 15625 active cells
    (34, 0.49, 5, 2),     # 4 or 2 lanes per cell
])
def test_lane_groups(prec, q, phi, nsel, sweeps):
    from paper_1211_1646_gb300 import hdmc
    w = W.fcc3(q, phi, 0.1, nselect=nsel)
    g = hdmc.System3(w.N, w.L, 1.0, w.d, nsel, 11, prec)
    r = O.System3(w.N, w.L, 1.0, w.d, nsel, 11, PREC[prec])
    g.sweep(sweeps)
    r.sweep(sweeps)
    _same(g, r)


def _column(K):
    """A dense crystal in a 4 x 4 x m column of wide cells (1.15 sigma): cells
    hold up to five spheres."""
    a = 4.6 / 3.0
    b = np.array([(0, 0, 0), (0.5, 0.5, 0), (0.5, 0, 0.5), (0, 0.5, 0.5)])
    i = np.stack(np.meshgrid(np.arange(K), np.arange(3), np.arange(3), indexing="ij"), -1).reshape(-1, 3)[:, ::-1]
    xyz = ((i[:, None, :] + b[None]) * a).reshape(-1, 3)
    return xyz + 0.25 * a, (4.6, 4.6, K * a)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("K", [8, 1500, 5600])
def test_crowded_cells(prec, K):
    # 4 cells per axis: a neighbour cell on either side may be the same cell
    from paper_1211_1646_gb300 import hdmc
    xyz, L = _column(K)
    g = hdmc.System3(len(xyz), L, 1.0, 0.12, 4, 3, prec, xyz=xyz)
    r = O.System3(len(xyz), L, 1.0, 0.12, 4, 3, PREC[prec], xyz=xyz)
    n = 40 if K == 8 else 4
    g.sweep(n)
    r.sweep(n)
    assert g.state()[1].max() >= 3
    _same(g, r)
