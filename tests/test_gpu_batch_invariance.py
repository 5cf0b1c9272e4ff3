"""FP64: a field's result does not depend on the batch it comes in.  The kernels of
the Legendre stage take 1 to 16 fields per CTA, as the batch and the order count
suggest; every width adds in the same order.  Orders of six segments, 129 pairs
(five groups of 32, one a single pair) and an equator row; 63 fields run 16 wide
with a ragged last CTA, the smaller batches 1, 2, 4 and 8 wide."""
import numpy as np
import pytest

import oracle
from paper_1202_6522_gb300 import synthetic

from _util import fp64_bound, normwise

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"
LMAX, NLAT, NPHI, FULL = 160, 257, 324, 63
NAMES = ["synth", "analys", "synth_adj", "analys_adj", "synth_vec", "analys_vec", "synth_vec_adj", "analys_vec_adj"]


@pytest.fixture(scope="module")
def setup():
    from paper_1202_6522_gb300 import SHT, build
    build.build()
    spec = [synthetic.spectrum(LMAX, batch=FULL, seed=s, power=1.5) for s in (1, 2)]
    grid = [synthetic.grid(NLAT, NPHI, batch=FULL, seed=s) for s in (3, 4)]
    return SHT(LMAX, LMAX, NLAT, NPHI, device=DEV), spec, grid


def _args(name, spec, grid):
    from_spec = name in ("synth", "analys_adj", "synth_vec", "analys_vec_adj")
    return (spec if from_spec else grid)[: 2 if "vec" in name else 1]


def _list(v):
    return list(v) if isinstance(v, tuple) else [v]


@pytest.mark.parametrize("name", NAMES)
def test_field_alone_and_in_batches(setup, name):
    sht, spec, grid = setup
    args = _args(name, spec, grid)
    dev = [torch.from_numpy(a).to(DEV) for a in args]
    full = _list(getattr(sht, name + "_")(*dev))
    for lo, hi in ((0, 1), (5, 7), (0, 3), (8, 16), (16, 32), (46, 63)):
        part = _list(getattr(sht, name + "_")(*[d[lo:hi].contiguous() for d in dev]))
        for p, f in zip(part, full):
            assert torch.equal(p, f[lo:hi]), (lo, hi)
    for b in (0, 62):
        ref = _list(getattr(oracle, name)(LMAX, LMAX, NLAT, NPHI, *[a[b:b + 1] for a in args]))
        for f, r in zip(full, ref):
            assert normwise(f[b].cpu().numpy(), np.asarray(r)[0]) <= fp64_bound(LMAX)


@pytest.mark.parametrize("lmax,nlat,nphi", [(255, 256, 512), (100, 101, 240)])
@pytest.mark.parametrize("name", NAMES[:4])
def test_tensor_core_field_alone_and_in_batches(name, lmax, nlat, nphi):
    """SHT_TC_F64: the contraction is exact in integers, the FFTs double-float."""
    from paper_1202_6522_gb300 import SHT
    sht = SHT(lmax, lmax, nlat, nphi, device=DEV, fp64_path="tc")
    spec = torch.from_numpy(synthetic.spectrum(lmax, batch=19, seed=1)).to(DEV)
    grid = torch.from_numpy(synthetic.grid(nlat, nphi, batch=19, seed=3)).to(DEV)
    x = _args(name, [spec], [grid])[0]
    full = getattr(sht, name + "_")(x)
    for lo, hi in ((0, 1), (2, 5), (8, 19)):
        assert torch.equal(getattr(sht, name + "_")(x[lo:hi].contiguous()), full[lo:hi])


@pytest.mark.parametrize("lmax", [63, 511])
@pytest.mark.parametrize("name", ["synth_", "analys_"])
def test_split_bf16_up_to_32_fields(name, lmax):
    """Split-bf16 products: up to 32 fields the sums of each product have columns of
    their own, and a field is the same in any such batch."""
    from paper_1202_6522_gb300 import SHT
    nlat, nphi = lmax + 1, 2 * (lmax + 1)
    sht = SHT(lmax, lmax, nlat, nphi, device=DEV, fp32_path="tc")
    if name == "synth_":
        x = torch.from_numpy(synthetic.spectrum(lmax, batch=32, seed=1).astype(np.complex64)).to(DEV)
    else:
        x = torch.from_numpy(synthetic.grid(nlat, nphi, batch=32, seed=3).astype(np.float32)).to(DEV)
    full = getattr(sht, name)(x)
    for lo, hi in ((0, 1), (0, 16), (15, 32), (3, 27)):
        assert torch.equal(getattr(sht, name)(x[lo:hi].contiguous()), full[lo:hi])
