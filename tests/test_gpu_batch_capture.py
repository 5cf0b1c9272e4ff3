"""Uneven batches captured by the caller into a graph of its own (relaxed
capture: the call allocates its staging): the replay computes what the call
would, also after other calls on the plan, and the plan stays usable."""
import numpy as np
import pytest

from paper_1202_6522_gb300 import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"
LMAX = [31, 9, 31, 63]


def test_graph_launch_stays_refused():
    from paper_1202_6522_gb300 import UnevenBatch, _capi as C, build
    build.build()
    ub = UnevenBatch(LMAX, use_graph=True, path="f32")
    specs = [torch.from_numpy(synthetic.spectrum(l, seed=i).astype(np.complex64)).to(DEV) for i, l in enumerate(LMAX)]
    grids = ub.synth_(specs)
    ref = [v.clone() for v in grids]
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="relaxed"):
        with pytest.raises(C.SHTError):
            ub.synth_(specs, out=grids)
        specs[0] + 1      # (a graph of something)
    for u, v in zip(ub.synth_(specs), ref):
        assert torch.equal(u, v)


@pytest.mark.parametrize("path", ["f32", "tc"])
def test_replay_after_other_calls(path):
    from paper_1202_6522_gb300 import UnevenBatch, build
    build.build()
    ub = UnevenBatch(LMAX, use_graph=False, path=path)
    specs = [[torch.from_numpy(synthetic.spectrum(l, seed=i + 9 * k).astype(np.complex64)).to(DEV)
              for i, l in enumerate(LMAX)] for k in range(2)]
    ref = [[v.clone() for v in ub.synth_(s)] for s in specs]
    back = [[v.clone() for v in ub.analys_(r)] for r in ref]
    grids = [torch.empty_like(v) for v in ref[0]]
    out = [torch.empty_like(v) for v in back[0]]
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="relaxed"):
        ub.synth_(specs[0], out=grids)
        ub.analys_(grids, out=out)
    other = ub.synth_(specs[1]), ub.analys_(ref[1])
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    for got, want in ((other[0], ref[1]), (other[1], back[1]), (grids, ref[0]), (out, back[0])):
        for u, v in zip(got, want):
            assert torch.equal(u, v)
