"""The automatic path of an uneven batch is chosen by the time of the form that
runs by default: graphs, in which the shapes' steps overlap."""
import numpy as np
import pytest

from paper_1202_6522_gb300 import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _pass_ms(ub, specs, grids, sout, gout):
    best = float("inf")
    for _ in range(5):
        for k in range(13):
            if k == 3:
                e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                e0.record()
            ub.synth_(specs, out=gout)
            ub.analys_(grids, out=sout)
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1) / 10)
    return best


def test_tuned_time_is_the_graphs():
    from paper_1202_6522_gb300 import UnevenBatch, build
    build.build()
    ls = synthetic.uneven_truncations(96)
    ub = UnevenBatch(ls, path="auto")
    specs = [torch.zeros(n, dtype=torch.complex64, device=DEV) for n in ub.nlm]
    grids = [torch.zeros(la, ph, device=DEV) for la, ph in zip(ub.nlat, ub.nphi)]
    sout, gout = [torch.empty_like(v) for v in specs], [torch.empty_like(v) for v in grids]
    ms = {}
    for graph in (True, False):
        tc = UnevenBatch(ls, path="tc", use_graph=graph)
        ms[graph] = _pass_ms(tc, specs, grids, sout, gout)
    assert abs(ub.tuned_ms["tc"] - ms[True]) < abs(ub.tuned_ms["tc"] - ms[False]), (ub.tuned_ms, ms)
