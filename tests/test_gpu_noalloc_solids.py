"""What lies at solid nodes and in the padding of the caller's buffers of lbm_step_noalloc is never read for a
result: no step writes there, so such memory may hold anything, NaN included.  The geometries have body-link
lists that do not fill a force group (128 links) and a solid, or fluid, node at (0, 0)."""
import numpy as np
import pytest

from paper_0904_4504_gb300 import lbm as L

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

DTYPE = {L.LBM_STORE_F64: torch.float64, L.LBM_STORE_F32: torch.float32, L.LBM_STORE_BF16: torch.bfloat16,
         L.LBM_STORE_F16: torch.float16}


def _corner(nx, ny):
    m = np.zeros((ny, nx), np.uint8)
    m[:5, :7] = 1
    m[ny - 4:, :3] = 2
    return m


GEOMETRY = {
    "plate": lambda nx, ny: dict(kind=L.LBM_GEOM_PLATE),
    "beam": lambda nx, ny: dict(kind=L.LBM_GEOM_BEAM, lx=9, ly=5),
    "corner": lambda nx, ny: dict(kind=L.LBM_GEOM_MASK, mask=_corner(nx, ny)),
}


@pytest.mark.parametrize("wall", [L.LBM_SCHEME_BOUNCEBACK, L.LBM_SCHEME_DIFFUSE], ids=["bounce", "diffuse"])
@pytest.mark.parametrize("storage", list(DTYPE), ids=["f64", "f32", "bf16", "f16"])
@pytest.mark.parametrize("geometry", GEOMETRY)
@pytest.mark.parametrize("Q,nx,ny", [(9, 45, 30), (37, 61, 41), (9, 520, 510)], ids=["q9", "q37", "q9-many"])
def test_values_at_solids_and_padding_do_not_matter(Q, nx, ny, geometry, storage, wall):
    geom = L.make_geometry(drive=L.LBM_DRIVE_WALL, u0=2e-3, eq_order=4 if Q == 37 else 2, storage=storage,
                           wall_scheme=wall, **GEOMETRY[geometry](nx, ny))
    sim = L.lbm_create(Q, nx, ny, 0.8, 0.05, geom)
    try:
        pitch = L.lbm_info(sim)["pitch"]
        solid = torch.ones((ny, pitch), dtype=torch.bool, device="cuda")
        solid[:, :nx] = torch.from_numpy(L.lbm_get_labels(sim) != 0).cuda()
        gen = torch.Generator(device="cuda").manual_seed(8)
        h = torch.randn((Q, ny, pitch), generator=gen, device="cuda").mul(1e-3).to(DTYPE[storage])
        runs = []
        for fill in (0.0, float("nan"), float("inf")):
            a, b = h.clone(), torch.full_like(h, fill)
            a[:, solid] = fill
            force = torch.zeros((2, 2), dtype=torch.float64, device="cuda")
            L.lbm_step_noalloc(sim, 3, a.data_ptr(), b.data_ptr(), force[0].data_ptr())
            L.lbm_step_noalloc(sim, 4, b.data_ptr(), a.data_ptr(), force[1].data_ptr())
            torch.cuda.synchronize()
            runs.append((a[:, ~solid].clone(), force))
        assert runs[0][0].isfinite().all() and runs[0][1].isfinite().all()
        for state, force in runs[1:]:
            assert torch.equal(state, runs[0][0]) and torch.equal(force, runs[0][1])
    finally:
        L.lbm_destroy(sim)
