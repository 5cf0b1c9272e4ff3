"""Uneven batches of more shapes than have an FFT launch of their own: launches
do not grow with the shapes beyond the contractions, and results equal the
per-field ones bit for bit, mixed-radix lengths included."""
import ctypes

import numpy as np
import pytest

from paper_1202_6522_gb300 import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _specs(ls):
    return [torch.from_numpy(synthetic.spectrum(l, seed=i).astype(np.complex64)).to(DEV) for i, l in enumerate(ls)]


def _graph_nodes(fn):
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g, capture_error_mode="relaxed"):
        fn()
    n = ctypes.c_size_t(0)
    assert ctypes.CDLL("libcudart.so.13").cudaGraphGetNodes(ctypes.c_void_p(g.raw_cuda_graph()), None,
                                                            ctypes.byref(n)) == 0
    return n.value


def test_one_copy_launch_for_all_shapes():
    """A tenth shape (an even number of coefficients: one contraction launch, no
    separate pass for its operand) adds one node per direction to the nine's."""
    from paper_1202_6522_gb300 import UnevenBatch, build
    build.build()
    nine = [5 + 3 * i for i in range(9)]
    nodes = []
    for ls in (nine, nine + [38]):
        assert (39 * 40 // 2) % 2 == 0
        ub = UnevenBatch(ls, use_graph=False, path="tc")
        specs = _specs(ls)
        grids, out = ub.synth_(specs), [torch.empty_like(v) for v in specs]
        ub.analys_(grids, out=out)
        torch.cuda.synchronize()
        nodes.append((_graph_nodes(lambda: ub.synth_(specs, out=grids)),
                      _graph_nodes(lambda: ub.analys_(grids, out=out))))
    assert [b - a for a, b in zip(*nodes)] == [1, 1]


# lmax, nphi: mixed radices on both sides of the lengths where the per-field FFTs
# change from radices up to 4 to radices up to 16 (256 in the analysis, 1024 in
# the synthesis), and a power of two
MIXED = [(30, 90), (47, 120), (63, 192), (95, 240), (100, 384), (120, 480), (127, 512), (140, 540), (60, 1080),
         (33, 1200), (20, 2160)]


@pytest.mark.parametrize("path", ["f32", "tc"])
def test_mixed_radix_equals_per_field(path):
    """(The CUDA-core analysis too: a warp sums a segment over the pairs in order
    in either form.)"""
    from paper_1202_6522_gb300 import SHT, UnevenBatch, build
    build.build()
    ls, nphis = [v[0] for v in MIXED], [v[1] for v in MIXED]
    ub = UnevenBatch(ls, nphi=nphis, path=path)
    specs = _specs(ls)
    grids = ub.synth_(specs)
    back = ub.analys_(grids)
    for l, n, s, g, a in zip(ls, nphis, specs, grids, back):
        one = SHT(l, l, l + 1, n, device=DEV, fp32_path=path)
        assert torch.equal(one.synth_(s[None])[0], g), (l, n)
        assert torch.equal(one.analys_(g[None])[0], a), (l, n)
