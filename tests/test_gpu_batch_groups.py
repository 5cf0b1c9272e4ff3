"""Uneven batches at the edge between one FFT launch per shape (up to eight
shapes, on branches of the graph) and the persistent FFT kernel (more), with
repeated shapes, an odd number of coefficients (copies that do not lie alike on
16 bytes), mixed-radix lengths and nphi = 4096; and calls that follow one another
without a host wait, on one stream and on two."""
import numpy as np
import pytest

from paper_1202_6522_gb300 import synthetic

import _bounds as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"

EIGHT = [(31, 32, 64), (5, 6, 12), (9, 12, 20), (31, 32, 64), (47, 48, 96), (20, 21, 4096), (63, 64, 128), (9, 12, 20),
         (15, 17, 32), (33, 34, 90)]
NINE = EIGHT + [(12, 13, 50)]


def _fields(shapes):
    specs = [synthetic.spectrum(l, seed=i).astype(np.complex64) for i, (l, _, _) in enumerate(shapes)]
    grids = [synthetic.grid(la, ph, seed=50 + i).astype(np.float32) for i, (_, la, ph) in enumerate(shapes)]
    return specs, grids


@pytest.mark.parametrize("path", ["f32", "tc"])
@pytest.mark.parametrize("use_graph", [True, False])
@pytest.mark.parametrize("shapes", [EIGHT, NINE], ids=["8shapes", "9shapes"])
def test_groups_match_oracle(shapes, use_graph, path):
    from paper_1202_6522_gb300 import UnevenBatch, build
    build.build()
    ub = UnevenBatch(*[list(v) for v in zip(*shapes)], use_graph=use_graph, path=path)
    specs, grids = _fields(shapes)
    got = ub.synth_([torch.from_numpy(s).to(DEV) for s in specs])
    back = ub.analys_([torch.from_numpy(g).to(DEV) for g in grids])
    torch.cuda.synchronize()
    for (l, la, ph), s, g, x, a in zip(shapes, specs, got, grids, back):
        B.assert_synth(g.cpu().numpy(), s.astype(np.complex128), l, l, la, ph, path, what=f"{path} group synth N{l}")
        B.assert_analys(a.cpu().numpy(), x.astype(np.float64), l, l, la, ph, path, what=f"{path} group analys N{l}")


@pytest.mark.parametrize("path", ["f32", "tc"])
def test_calls_without_host_waits(path):
    """Eight calls in a row, alternating direction, inputs and then streams: each
    result equals that of the same call made alone."""
    from paper_1202_6522_gb300 import UnevenBatch, build
    build.build()
    ub = UnevenBatch(*[list(v) for v in zip(*EIGHT)], path=path)
    specs, grids = _fields(EIGHT)
    sp = [[torch.from_numpy(s * (k + 1)).to(DEV) for s in specs] for k in range(4)]
    gr = [[torch.from_numpy(g * (k + 1)).to(DEV) for g in grids] for k in range(4)]
    alone = []
    for k in range(4):
        alone.append(ub.synth_(sp[k]))
        torch.cuda.synchronize()
        alone.append(ub.analys_(gr[k]))
        torch.cuda.synchronize()
    for streams in ([torch.cuda.current_stream()] * 2, [torch.cuda.Stream(), torch.cuda.Stream()]):
        torch.cuda.synchronize()
        got = []
        for k in range(4):
            with torch.cuda.stream(streams[0]):
                got.append(ub.synth_(sp[k]))
            with torch.cuda.stream(streams[1]):
                got.append(ub.analys_(gr[k]))
        torch.cuda.synchronize()
        for a, g in zip(alone, got):
            for u, v in zip(a, g):
                assert torch.equal(u, v)
