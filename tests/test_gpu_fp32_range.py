"""FP32 analyses of data of small magnitude: scaled by a power of two, the data
give the result scaled by the same power.  High orders start segments from
states far below the range of their later values; the terms P_n^m times fold of
such a segment are ordinary FP32 numbers however small the data are.

Tolerance: 2^-80 times O(1) data.  Scaling by a power of two commutes with every
rounding except that of a result below 2^-126, which is off by at most 2^-150,
2^-70 of the unscaled data.  An output is reached by fewer than 2^14 operations
(two FFTs of length 1024, 512 pairs, 32 degrees of recurrence), each amplified
by at most 2^24 (order 1023 of the vector terms, 1 / sin(theta), |P| < 32): 2^-32."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"

N, SCALE, TOL = 1023, 2.0 ** -80, 2.0 ** -32


@pytest.fixture(scope="module")
def setup():
    from paper_1202_6522_gb300 import SHT, build
    build.build()
    gen = torch.Generator(device=DEV).manual_seed(1)
    grids = [torch.randn(3, N + 1, 2 * N + 2, generator=gen, device=DEV) for _ in range(2)]
    return SHT(N, N, N + 1, 2 * N + 2, device=DEV), grids


@pytest.mark.parametrize("batch", [1, 3])
@pytest.mark.parametrize("name", ["analys_", "synth_adj_", "analys_vec_", "synth_vec_adj_"])
def test_small_data(setup, name, batch):
    sht, grids = setup
    args = [g[:batch].contiguous() for g in (grids if "vec" in name else grids[:1])]
    ref, got = (getattr(sht, name)(*[a * f for a in args]) for f in (1.0, SCALE))
    for r, g in zip(*(v if isinstance(v, tuple) else (v,) for v in (ref, got))):
        assert float((g.to(torch.complex128) / SCALE - r).abs().max()) <= TOL


def test_small_data_uneven_batch():
    from paper_1202_6522_gb300 import UnevenBatch
    gen = torch.Generator(device=DEV).manual_seed(2)
    ub = UnevenBatch([N, 63], path="f32")
    grids = [torch.randn(n + 1, 2 * n + 2, generator=gen, device=DEV) for n in (N, 63)]
    ref = [v.clone() for v in ub.analys_(grids)]
    got = ub.analys_([g * SCALE for g in grids])
    for r, g in zip(ref, got):
        assert float((g.to(torch.complex128) / SCALE - r).abs().max()) <= TOL
