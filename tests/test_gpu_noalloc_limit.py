"""lbm_step_noalloc accepts up to LBM_NOALLOC_MAX_SLOTS (8192) tiles with body links.  The kernels that lbm_create
chooses by itself for 16-bit D2Q37 and large FP32 D2Q9 grids have tiles of one row or two, which must not make
a tall body too large for it."""
import pytest

from paper_0904_4504_gb300 import lbm as L

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

DTYPE = {L.LBM_STORE_F32: torch.float32, L.LBM_STORE_F16: torch.float16}


def _sim(Q, nx, ny, lx, ly, storage):
    geom = L.make_geometry(kind=L.LBM_GEOM_BEAM, lx=lx, ly=ly, drive=L.LBM_DRIVE_WALL, u0=2e-3, eq_order=4 if Q == 37 else 2,
                           storage=storage)
    return L.lbm_create(Q, nx, ny, 0.8, 0.05, geom)


# 2064, 2064 and about 8000 tiles of 32 x 4 nodes hold body links (of the pairs' own 64 x 1: 8212)
@pytest.mark.parametrize("Q,nx,ny,lx,ly,storage,variant", [
    (37, 128, 4200, 70, 4100, L.LBM_STORE_F16, 31),
    (37, 640, 4200, 70, 4100, L.LBM_STORE_F16, 32),
    (9, 100, 17000, 70, 16000, L.LBM_STORE_F32, 30)], ids=["pairs", "staged-pairs", "q9"])
def test_tall_bodies_on_the_default_kernels(Q, nx, ny, lx, ly, storage, variant):
    sim, plain = _sim(Q, nx, ny, lx, ly, storage), _sim(Q, nx, ny, lx, ly, storage)
    try:
        info = L.lbm_info(sim)
        assert info["variant"] == variant
        L.lbm_set_tile(plain, 32, 4)
        gen = torch.Generator(device="cuda").manual_seed(5)
        h = torch.randn(Q * ny * info["pitch"], generator=gen, device="cuda").mul(1e-3).to(DTYPE[storage])
        got = []
        for handle in (plain, sim):
            out, force = torch.zeros_like(h), torch.zeros(2, dtype=torch.float64, device="cuda")
            L.lbm_step_noalloc(handle, 3, h.data_ptr(), out.data_ptr(), force.data_ptr())
            torch.cuda.synchronize()
            got.append((out, force))
        assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
        assert got[0][1].isfinite().all() and got[0][1].abs().max() > 0
    finally:
        L.lbm_destroy(sim)
        L.lbm_destroy(plain)


def test_the_tile_shape_decides_where_it_is_the_callers():
    """On 32 x 1 tiles the beam has 2 x 4106 of them, on 32 x 4 a quarter: refused, then accepted."""
    sim = _sim(37, 128, 4200, 70, 4100, L.LBM_STORE_F32)
    try:
        n = 37 * 4200 * L.lbm_info(sim)["pitch"]
        a, b = torch.zeros(n, device="cuda"), torch.zeros(n, device="cuda")
        force = torch.zeros(2, dtype=torch.float64, device="cuda")
        for tile, fits in (((32, 1), False), ((32, 4), True), ((64, 1), False), ((128, 4), True)):
            L.lbm_set_tile(sim, *tile)
            if fits:
                L.lbm_step_noalloc(sim, 0, a.data_ptr(), b.data_ptr(), force.data_ptr())
                continue
            with pytest.raises(L.LbmError) as e:
                L.lbm_step_noalloc(sim, 0, a.data_ptr(), b.data_ptr(), force.data_ptr())
            assert e.value.code == L.LBM_ERANGE
        torch.cuda.synchronize()
    finally:
        L.lbm_destroy(sim)
