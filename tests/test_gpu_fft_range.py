"""Analyses of constant fields near the top of the number range, through the tile
FFTs (mixed radices; FP64 and lengths above 2048 at any radix): nothing on the
way needs more than the sum of a row and its mirror row, 2 nphi F, here 0.6 of
the largest number (four times nphi F would exceed it).  FP64 with few degrees:
its Legendre sums run on P divided by a power of the recurrence's growth."""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


F32, F64 = torch.float32, torch.float64


@pytest.mark.parametrize("dtype,lmax,nphi", [(F32, 5, 12), (F32, 40, 90), (F32, 100, 384), (F32, 60, 540),
                                             (F32, 31, 4096), (F32, 7, 2160), (F64, 5, 12), (F64, 7, 256),
                                             (F64, 7, 2160), (F64, 7, 4096)])
def test_constant_field(dtype, lmax, nphi):
    from paper_1202_6522_gb300 import SHT, build
    build.build()
    sht = SHT(lmax, lmax, lmax + 1, nphi, device=DEV)
    F = 0.6 * torch.finfo(dtype).max / (2 * nphi)
    got = sht.analys_(torch.full((1, lmax + 1, nphi), F, dtype=dtype, device=DEV))[0] / F
    # f_0^0 = sqrt(4 pi) F, to 2 log2(nphi) roundings of the FFT and lmax + 1 of the sum
    tol = math.sqrt(4 * math.pi) * (2 * math.log2(nphi) + lmax + 1) * torch.finfo(dtype).eps
    assert abs(complex(got[0]) - math.sqrt(4 * math.pi)) <= tol
    assert torch.isfinite(torch.view_as_real(got)).all()
