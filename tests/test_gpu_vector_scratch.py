"""Memory of the FP64 vector transforms: they ask for nothing beyond the two
intermediates of the scratch, so that a call whose scratch an earlier call left
can be captured, and sht_reserve holds no more than that."""
import pytest

from paper_1202_6522_gb300 import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def lib():
    from paper_1202_6522_gb300 import build
    build.build()
    import paper_1202_6522_gb300
    return paper_1202_6522_gb300


def _inputs(lmax, nlat, nphi, batch):
    spec = [torch.from_numpy(synthetic.spectrum(lmax, batch=batch, seed=s, power=1.5)).to(DEV) for s in (1, 2)]
    grid = [torch.from_numpy(synthetic.grid(nlat, nphi, batch=batch, seed=s)).to(DEV) for s in (3, 4)]
    return {"synth_vec_": spec, "analys_vec_": grid, "synth_vec_adj_": grid, "analys_vec_adj_": spec}


def _captured(fn):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = fn()
    g.replay()
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("name", ["synth_vec_", "analys_vec_", "synth_vec_adj_", "analys_vec_adj_"])
@pytest.mark.parametrize("lmax,nlat,nphi,batch", [(63, 64, 128, 2), (0, 1, 2, 3), (33, 41, 90, 5)])
def test_captured_after_a_scalar_call(lib, name, lmax, nlat, nphi, batch):
    """A scalar call of twice as many fields leaves the scratch a vector call takes."""
    sht = lib.SHT(lmax, lmax, nlat, nphi, device=DEV)
    sht.synth_(torch.from_numpy(synthetic.spectrum(lmax, batch=2 * batch, seed=0)).to(DEV))
    args = _inputs(lmax, nlat, nphi, batch)[name]
    got = _captured(lambda: getattr(sht, name)(*args))
    for g, r in zip(got, getattr(sht, name)(*args)):
        assert torch.equal(g, r)


def test_reserve_holds_the_intermediates_only(lib):
    from paper_1202_6522_gb300 import _capi as C
    lmax, nlat, nphi, batch = 255, 256, 512, 256
    sht = lib.SHT(lmax, lmax, nlat, nphi, device=DEV)
    C.sht_reserve(sht._h, 1, C.SHT_F64)   # the tables
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    C.sht_reserve(sht._h, batch, C.SHT_F64)
    inter = batch * (lmax + 1) * (nlat // 2) * 4 * 8
    assert before - torch.cuda.mem_get_info()[0] <= 2 * inter * (1 + 1 / nlat) + (4 << 20)
