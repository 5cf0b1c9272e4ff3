"""FP32 Legendre stage on the CUDA cores at the sizes where its split changes:
orders whose degrees end on a 32-degree segment or one past it, segment counts
around the four a CTA takes, pair counts at the edges of 32 and 64 and of the
ring of four, field counts at the edges of the widths 1, 2 and 4, few orders
and an equator row.  Every direction, scalar and vector, and its adjoint,
within the bounds derived from the arithmetic."""
import numpy as np
import pytest

import oracle
from paper_1202_6522_gb300 import synthetic

import _bounds as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"

# (lmax, mmax, nlat, nphi, batch)
SHAPES = [
    (1, 1, 2, 4, 2),
    (31, 31, 32, 64, 1),       # order 0 fills one segment
    (32, 32, 65, 72, 3),       # one degree in a second one, 33 pairs, equator row
    (63, 63, 128, 128, 5),     # 64 pairs
    (127, 40, 129, 96, 2),     # four segments, 65 pairs
    (128, 128, 257, 270, 1),   # a fifth segment, 129 pairs (five groups)
    (200, 5, 320, 16, 9),      # few orders, many fields, 160 pairs
]


def _np(t):
    return t.detach().cpu().numpy().astype(np.complex128 if t.is_complex() else np.float64)


@pytest.mark.parametrize("lmax,mmax,nlat,nphi,batch", SHAPES)
def test_fp32_legendre_edges(lmax, mmax, nlat, nphi, batch):
    from paper_1202_6522_gb300 import SHT, build
    build.build()
    sht = SHT(lmax, mmax, nlat, nphi, device=DEV)
    a, b = (synthetic.spectrum(lmax, mmax, batch=batch, seed=s, power=1.5).astype(np.complex64) for s in (5, 6))
    x, y = (synthetic.grid(nlat, nphi, batch=batch, seed=s).astype(np.float32) for s in (7, 8))
    da, db, dx, dy = (torch.from_numpy(v).to(DEV) for v in (a, b, x, y))
    a, b, x, y = (v.astype(np.complex128 if v.dtype.kind == "c" else np.float64) for v in (a, b, x, y))
    size = (lmax, mmax, nlat, nphi)
    B.assert_synth(_np(sht.synth_(da)), a, *size, "f32", what="f32 synth")
    B.assert_analys(_np(sht.analys_(dx)), x, *size, "f32", what="f32 analys")
    B.check_scalar_adjoints(_np(sht.synth_adj_(dx)), _np(sht.analys_adj_(da)), x, a, *size, "f32", "f32")
    vt, vp = sht.synth_vec_(da, db)
    S, T = sht.analys_vec_(dx, dy)
    rt, rp = oracle.synth_vec(*size, a, b)
    rS, rT = oracle.analys_vec(*size, x, y)
    B.check_vector(_np(vt), _np(vp), rt, rp, a, b, _np(S), _np(T), rS, rT, x, y, *size, "f32", "f32")
    S, T = sht.synth_vec_adj_(dx, dy)
    ht, hp = sht.analys_vec_adj_(da, db)
    rS, rT = oracle.synth_vec_adj(*size, x, y)
    rt, rp = oracle.analys_vec_adj(*size, a, b)
    B.check_vector_adjoints(_np(S), _np(T), rS, rT, x, y, _np(ht), _np(hp), rt, rp, a, b, *size, "f32", "f32")
