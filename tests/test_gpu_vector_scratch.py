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
@pytest.mark.parametrize("lmax,nlat,nphi,batch", [(63, 64, 128, 2), (0, 1, 2, 3), (33, 41, 90, 5), (40, 41, 96, 70)])
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


@pytest.mark.parametrize("name", ["synth_vec_", "analys_vec_", "synth_vec_adj_", "analys_vec_adj_"])
@pytest.mark.parametrize("lmax,mmax,mres,nlat,nphi,batch", [(63, 63, 1, 64, 128, 2), (0, 0, 1, 1, 2, 1),
                                                            (31, 31, 1, 33, 64, 9), (340, 340, 1, 341, 720, 1),
                                                            (95, 31, 3, 96, 80, 3)])
def test_captured_on_a_plan_without_tables(lib, name, lmax, mmax, mres, nlat, nphi, batch):
    """Tables cannot be built under capture.  A plan whose scratch was left by a
    call in another mode runs without them, to the same bits."""
    from paper_1202_6522_gb300 import _capi as C
    gen = torch.Generator(device=DEV).manual_seed(3)
    sht = lib.SHT(lmax, mmax, nlat, nphi, device=DEV, mres=mres)
    if "synth_vec_" == name or "analys_vec_adj_" == name:
        args = [torch.randn(batch, sht.nlm, dtype=torch.complex128, generator=gen, device=DEV) for _ in range(2)]
    else:
        args = [torch.randn(batch, nlat, nphi, dtype=torch.float64, generator=gen, device=DEV) for _ in range(2)]
    C.sht_reserve(sht._h, 2 * batch, C.SHT_F32)   # as many bytes as two FP64 intermediates of `batch` fields
    got = _captured(lambda: getattr(sht, name)(*args))
    for g, r in zip(got, getattr(sht, name)(*args)):
        assert torch.equal(g, r)


@pytest.mark.parametrize("reserve", [False, True])
def test_tensor_core_plan_captures_vector_calls(lib, reserve):
    """A plan in SHT_TC_F64, whose vector transforms run SHT_F64."""
    from paper_1202_6522_gb300 import _capi as C
    lmax, nlat, nphi, batch = 63, 64, 128, 2
    sht = lib.SHT(lmax, lmax, nlat, nphi, device=DEV, fp64_path="tc")
    args = _inputs(lmax, nlat, nphi, batch)
    if reserve:
        C.sht_reserve(sht._h, batch, C.SHT_TC_F64)
    else:
        sht.synth_(args["synth_vec_"][0])
    for name, a in args.items():
        got = _captured(lambda: getattr(sht, name)(*a))
        for g, r in zip(got, getattr(sht, name)(*a)):
            assert torch.equal(g, r)


def test_no_memory_for_the_tables(lib):
    """Tables of 217 MB (lmax = 1023: 20 B per pair and 32 degrees, 40 B per
    coefficient) where 160 MiB are left: the call runs without them, to the same bits."""
    lmax, nlat, nphi = 1023, 1024, 2048
    gen = torch.Generator(device=DEV).manual_seed(3)
    grid = [torch.randn(1, nlat, nphi, dtype=torch.float64, generator=gen, device=DEV) for _ in range(2)]
    sht = lib.SHT(lmax, lmax, nlat, nphi, device=DEV)
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - (160 << 20), dtype=torch.uint8, device=DEV)
    got = sht.analys_vec_(*grid)
    torch.cuda.synchronize()
    del hog
    torch.cuda.empty_cache()
    for g, r in zip(got, sht.analys_vec_(*grid)):
        assert torch.equal(g, r)
