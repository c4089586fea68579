"""Sphere sweeps on a stream that the caller records (the launches themselves are
recorded), and parameters changed after sweeps were recorded into graphs: the
oracle's chain, bit for bit."""
import numpy as np
import pytest

import oracle as O
from paper_1211_1646_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PREC = {"fp64": O.FP64, "fp32": O.FP32}


def _same(g, r):
    lg, cg = g.state()
    lr, cr = r.state()
    assert np.array_equal(cg, cr)
    assert np.array_equal(lg, lr)
    assert np.array_equal(g.counters(), r.counters())
    assert np.array_equal(g.origin(), r.origin())


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1211_1646_gb300 import build
    build.build()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("sweeps", [3, 70])   # within and beyond one table of draws
def test_recorded_by_the_caller(prec, sweeps):
    import torch
    from paper_1211_1646_gb300 import hdmc
    w = W.fcc3(8, 0.45, 0.1)
    stream = torch.cuda.Stream()
    g = hdmc.System3(w.N, w.L, 1.0, w.d, 4, 11, prec, stream=stream.cuda_stream)
    r = O.System3(w.N, w.L, 1.0, w.d, 4, 11, PREC[prec])
    g.sweep(5)
    r.sweep(5)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        g.sweep(sweeps)
    with torch.cuda.stream(stream):
        graph.replay()
    r.sweep(sweeps)
    _same(g, r)
    g.sweep(2)
    r.sweep(2)
    _same(g, r)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_parameters_changed_after_recording(prec):
    from paper_1211_1646_gb300 import hdmc
    w = W.fcc3(8, 0.45, 0.1)
    g = hdmc.System3(w.N, w.L, 1.0, 0.1, 4, 11, prec)
    r = O.System3(w.N, w.L, 1.0, 0.1, 4, 11, PREC[prec])
    for d, shuffle in ((0.1, True), (0.05, True), (0.05, False), (0.2, True)):
        hdmc.hdmc3_set_move_size(g.h, d)
        hdmc.hdmc3_set_balance(g.h, shuffle, True)
        r.set_move_size(d)
        r.set_balance(shuffle, True)
        for n in (1, 7, 32, 1):
            g.sweep(n)
            r.sweep(n)
        _same(g, r)
