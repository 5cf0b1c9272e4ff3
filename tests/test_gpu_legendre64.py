"""FP64 Legendre stage on the CUDA cores at the sizes where its split changes:
orders whose degrees end on a 32-degree segment or one past it (the vector
transforms run one degree further), pair counts at the edges of 32 and of 128,
field counts at the edges of the widths 1 .. 16, strided orders, and an
equator row.  Every direction, scalar and vector, and its adjoint, against the
oracle."""
import numpy as np
import pytest

import oracle
from paper_1202_6522_gb300 import synthetic

from _util import fp64_bound, normwise

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"

# (lmax, mmax, nlat, nphi, batch)
SHAPES = [
    (0, 0, 1, 2, 1),
    (1, 1, 2, 4, 2),
    (31, 31, 32, 64, 1),       # order 0 fills one segment
    (32, 32, 33, 72, 3),       # one degree in a second one, equator row
    (63, 63, 64, 128, 1),      # 32 pairs
    (62, 62, 65, 128, 2),      # 33 pairs
    (64, 64, 130, 144, 9),     # 65 pairs
    (95, 40, 256, 96, 5),      # 128 pairs
    (95, 95, 257, 192, 17),    # 129 pairs, a field beyond a width of 16
    (127, 127, 192, 384, 1),
    (160, 9, 161, 20, 33),     # few orders, many fields
]


@pytest.mark.parametrize("lmax,mmax,nlat,nphi,batch", SHAPES)
def test_fp64_legendre_edges(lmax, mmax, nlat, nphi, batch):
    from paper_1202_6522_gb300 import SHT, build
    build.build()
    sht = SHT(lmax, mmax, nlat, nphi, device=DEV)
    dev = lambda v: torch.from_numpy(v).to(DEV)  # noqa: E731
    a, b = (synthetic.spectrum(lmax, mmax, batch=batch, seed=s, power=1.5) for s in (5, 6))
    x, y = (synthetic.grid(nlat, nphi, batch=batch, seed=s) for s in (7, 8))
    size = (lmax, mmax, nlat, nphi)
    pairs = [([sht.synth_(dev(a))], [oracle.synth(*size, a)]),
             ([sht.analys_(dev(x))], [oracle.analys(*size, x)]),
             ([sht.synth_adj_(dev(x))], [oracle.synth_adj(*size, x)]),
             ([sht.analys_adj_(dev(a))], [oracle.analys_adj(*size, a)]),
             (sht.synth_vec_(dev(a), dev(b)), oracle.synth_vec(*size, a, b)),
             (sht.analys_vec_(dev(x), dev(y)), oracle.analys_vec(*size, x, y)),
             (sht.synth_vec_adj_(dev(x), dev(y)), oracle.synth_vec_adj(*size, x, y)),
             (sht.analys_vec_adj_(dev(a), dev(b)), oracle.analys_vec_adj(*size, a, b))]
    for got, ref in pairs:
        scale = max(np.abs(r).max() for r in ref)
        for g, r in zip(got, ref):
            err = np.abs(g.cpu().numpy() - r).max()
            assert err <= fp64_bound(lmax) * scale


@pytest.mark.parametrize("lmax,mres,mmax", [(64, 2, 32), (95, 3, 31), (96, 5, 19)])
def test_fp64_vector_strided_orders(lmax, mres, mmax):
    """An m-stride plan's vector transform equals the full plan's on the same
    orders (spectra zero elsewhere), longitudes of one sector."""
    from paper_1202_6522_gb300 import SHT, build
    build.build()
    nlat, nphi = lmax + 1, 80
    one = SHT(lmax, mmax, nlat, nphi, device=DEV, mres=mres)
    full = SHT(lmax, mmax * mres, nlat, nphi * mres, device=DEV)
    rng = np.random.default_rng(1)
    s, t = (np.zeros((2, one.nlm), dtype=complex) for _ in range(2))
    fs, ft = (np.zeros((2, full.nlm), dtype=complex) for _ in range(2))
    for k in range(mmax + 1):
        for n in range(k * mres, lmax + 1):
            for v, f in ((s, fs), (t, ft)):
                z = rng.standard_normal(2) + 1j * rng.standard_normal(2) * (k > 0)
                v[:, one.lm_index(n, k * mres)] = z / (n + 1)
                f[:, full.lm_index(n, k * mres)] = z / (n + 1)
    dev = lambda v: torch.from_numpy(v).to(DEV)  # noqa: E731
    got = one.synth_vec_(dev(s), dev(t))
    ref = full.synth_vec_(dev(fs), dev(ft))
    for g, r in zip(got, ref):
        assert normwise(g.cpu().numpy(), r.cpu().numpy()[..., :nphi]) < 1e-12
    back = one.analys_vec_(*got)
    for g, r in zip(back, (s, t)):
        r = r.copy()
        r[:, 0] = 0        # the degree 0 has no vector part
        assert normwise(g.cpu().numpy(), r) < 1e-12


def test_fp64_vector_graph_outlives_a_larger_call():
    """A captured vector transform replays after a call with more fields, whose
    intermediates fit the scratch that a scalar call left, took larger spectra."""
    from paper_1202_6522_gb300 import SHT, build
    build.build()
    lmax, nlat, nphi = 40, 48, 96
    sht = SHT(lmax, lmax, nlat, nphi, device=DEV)
    dev = lambda v: torch.from_numpy(v).to(DEV)  # noqa: E731
    a, b = (synthetic.spectrum(lmax, lmax, batch=9, seed=s, power=1.5) for s in (5, 6))
    sht.synth_(dev(synthetic.spectrum(lmax, lmax, batch=64, seed=1, power=1.5)))
    S, T = dev(a[:2]), dev(b[:2])
    ref = [v.clone() for v in sht.synth_vec_(S, T)]
    out = [torch.empty_like(v) for v in ref]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        for o, v in zip(out, sht.synth_vec_(S, T)):
            o.copy_(v)
    sht.synth_vec_(dev(a), dev(b))
    g.replay()
    torch.cuda.synchronize()
    for o, r in zip(out, ref):
        assert torch.equal(o, r)
