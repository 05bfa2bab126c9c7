"""lbm_step_noalloc runs the simulation's own kernel where the caller's buffers are aligned for it and the
plain one elsewhere: both give the plain kernel's bits, and only fluid nodes are written."""
import numpy as np
import pytest

from paper_0904_4504_gb300 import lbm as L

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

DTYPE = {L.LBM_STORE_F64: torch.float64, L.LBM_STORE_F32: torch.float32, L.LBM_STORE_BF16: torch.bfloat16,
         L.LBM_STORE_F16: torch.float16}


@pytest.mark.parametrize("Q,nx,ny,st,wall", [
    (37, 131, 61, L.LBM_STORE_F16, 0), (37, 2048, 680, L.LBM_STORE_F16, 0), (37, 47, 80, L.LBM_STORE_BF16, 0),
    (37, 90, 61, L.LBM_STORE_F32, 0), (37, 90, 61, L.LBM_STORE_F64, 0), (37, 90, 61, L.LBM_STORE_F32, 1),
    (9, 530, 521, L.LBM_STORE_F32, 0), (9, 531, 257, L.LBM_STORE_F16, 0), (9, 61, 45, L.LBM_STORE_F64, 0)],
    ids=["q37-f16", "q37-f16-staged", "q37-bf16-narrow", "q37-f32", "q37-f64", "q37-f32-diffuse", "q9-f32", "q9-f16",
         "q9-f64"])
def test_same_bits_for_any_alignment(Q, nx, ny, st, wall):
    geom = L.make_geometry(kind=L.LBM_GEOM_BEAM, lx=13, ly=11, drive=L.LBM_DRIVE_WALL, u0=2e-3,
                           eq_order=4 if Q == 37 else 2, storage=st, wall_scheme=wall)
    sim = L.lbm_create(Q, nx, ny, 0.8, 0.05, geom)
    plain = L.lbm_create(Q, nx, ny, 0.8, 0.05, geom)
    L.lbm_set_tile(plain, 32, 4)
    try:
        pitch, n = L.lbm_info(sim)["pitch"], Q * ny * L.lbm_info(sim)["pitch"]
        gen = torch.Generator(device="cuda").manual_seed(4)
        h = torch.randn(n, generator=gen, device="cuda").to(DTYPE[st])
        solid = torch.zeros((ny, pitch), dtype=torch.bool, device="cuda")
        solid[:, nx:] = True
        solid[:, :nx] |= torch.from_numpy(L.lbm_get_labels(sim) != 0).cuda()
        want = None
        for handle, offset in ((plain, 0), (sim, 0), (sim, 1), (sim, 2)):
            a = torch.empty(n + 2, dtype=DTYPE[st], device="cuda")
            b = torch.full_like(a, 7.0)
            a[offset:offset + n] = h
            force = torch.zeros(2, dtype=torch.float64, device="cuda")
            es = a.element_size()
            L.lbm_step_noalloc(handle, 3, a.data_ptr() + offset * es, b.data_ptr() + offset * es, force.data_ptr())
            torch.cuda.synchronize()
            got = b[offset:offset + n].view(Q, ny, pitch)
            assert (got[:, solid] == 7.0).all() and (b[:offset] == 7.0).all() and (b[offset + n:] == 7.0).all()
            if want is None:
                want = got.clone(), force.clone()
            assert torch.equal(got, want[0]) and torch.equal(force, want[1]), offset
    finally:
        L.lbm_destroy(sim)
        L.lbm_destroy(plain)
