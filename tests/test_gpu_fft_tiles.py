"""FP64 longitude FFTs at the lengths where the tile changes: 4 or 16 values per
thread (H = nphi / 2 up to 1024 or above), radix 3 and 5 passes that leave
threads without an item, one latitude pair per CTA (few rows) or several (many
rows), an odd number of latitudes (equator row), and the highest order m next
to H, whose partner position H - m shares its product."""
import numpy as np
import pytest

import oracle
from paper_1202_6522_gb300 import synthetic

from _util import fp64_bound, normwise

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"

# (lmax, nlat, nphi, batch)
SHAPES = [
    (0, 1, 2, 1),            # H = 1
    (1, 3, 4, 2),            # H = 2
    (2, 5, 6, 3),            # H = 3: the order next to H
    (4, 5, 10, 1),           # H = 5: more threads than items
    (7, 9, 30, 300),         # H = 15, several pairs per CTA
    (15, 17, 32, 700),       # H = 16, several pairs per CTA
    (31, 32, 64, 1),         # H = 32, one pair per CTA
    (20, 21, 2000, 2),       # H = 1000
    (20, 21, 2048, 2),       # H = 1024, the longest with 4 values per thread
    (20, 21, 2160, 2),       # H = 1080, 16 values per thread
    (20, 21, 4096, 1),       # H = 2048
]


@pytest.mark.parametrize("lmax,nlat,nphi,batch", SHAPES)
def test_fp64_fft_tile_edges(lmax, nlat, nphi, batch):
    from paper_1202_6522_gb300 import SHT, build
    build.build()
    sht = SHT(lmax, lmax, nlat, nphi, device=DEV)
    a = synthetic.spectrum(lmax, batch=batch, seed=3)
    x = synthetic.grid(nlat, nphi, batch=batch, seed=4)
    at, xt = torch.from_numpy(a).to(DEV), torch.from_numpy(x).to(DEV)
    got = [sht.synth_(at), sht.analys_(xt), sht.synth_adj_(xt), sht.analys_adj_(at)]
    ref = [oracle.synth(lmax, lmax, nlat, nphi, a), oracle.analys(lmax, lmax, nlat, nphi, x),
           oracle.synth_adj(lmax, lmax, nlat, nphi, x), oracle.analys_adj(lmax, lmax, nlat, nphi, a)]
    for g, r in zip(got, ref):
        assert normwise(g.cpu().numpy(), r) < fp64_bound(lmax)


# (lmax, nlat, nphi, batch): the FP64-accurate tensor-core mode's double-float
# FFTs and the FP32 mixed-radix ones, where their values per thread change
MIXED = [
    (15, 17, 36, 1),         # H = 18
    (15, 17, 500, 3),        # H = 250
    (15, 17, 540, 3),        # H = 270: FP32 analysis with 16 values
    (15, 17, 2000, 2),       # H = 1000
    (15, 17, 2160, 2),       # H = 1080: 16 values throughout
    (15, 17, 1024, 2),       # H = 512, few rows
    (15, 17, 1024, 160),     # H = 512, many rows
    (15, 17, 2048, 1),       # H = 1024, few rows
    (15, 17, 2048, 64),      # H = 1024, many rows
]


@pytest.mark.parametrize("lmax,nlat,nphi,batch", MIXED)
def test_double_float_and_fp32_tiles(lmax, nlat, nphi, batch):
    import _bounds as B
    from paper_1202_6522_gb300 import SHT, build
    build.build()
    size = (lmax, lmax, nlat, nphi)
    a = synthetic.spectrum(lmax, batch=batch, seed=3)
    x = synthetic.grid(nlat, nphi, batch=batch, seed=4)
    tc = SHT(*size, device=DEV, fp64_path="tc")
    assert normwise(tc.synth_(torch.from_numpy(a).to(DEV)).cpu().numpy(), oracle.synth(*size, a)) < fp64_bound(lmax)
    assert normwise(tc.analys_(torch.from_numpy(x).to(DEV)).cpu().numpy(), oracle.analys(*size, x)) < fp64_bound(lmax)
    a, x = a[:4].astype(np.complex64), x[:4].astype(np.float32)
    f32 = SHT(*size, device=DEV)
    B.assert_synth(f32.synth_(torch.from_numpy(a).to(DEV)).cpu().numpy(), a.astype(np.complex128), *size, "f32")
    B.assert_analys(f32.analys_(torch.from_numpy(x).to(DEV)).cpu().numpy(), x.astype(np.float64), *size, "f32")
