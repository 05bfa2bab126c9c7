"""The kernel that lbm_create and a batch choose by themselves, around the lines of the rules.  Regularized D2Q37
with 16-bit storage: few columns that would leave half a block idle, small grids, and where staging pays; D2Q9:
narrow and small grids."""
import pytest

from paper_0904_4504_gb300 import lbm as L

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


def _kw(storage, collision):
    return dict(kind=L.LBM_GEOM_NONE, u0=1e-3, eq_order=4, storage=storage, collision=collision)


@pytest.mark.parametrize("storage", [L.LBM_STORE_F16, L.LBM_STORE_BF16], ids=["f16", "bf16"])
@pytest.mark.parametrize("nx,ny,alone,batch", [
    (24, 24, 2, 32), (32, 9000, 2, 2), (33, 9000, 31, 31), (64, 64, 2, 32), (65, 4000, 2, 2), (96, 4000, 2, 2),
    (97, 4000, 31, 31), (160, 2000, 2, 2), (161, 2000, 31, 31), (300, 599, 31, 32), (300, 600, 31, 31), (447, 894, 31, 31),
    (448, 357, 2, 32), (448, 896, 31, 32), (512, 312, 2, 32), (512, 313, 31, 32), (639, 2200, 31, 32), (640, 2200, 32, 32),
    (1024, 1024, 31, 32)])
def test_pairs_by_the_grids_sides(nx, ny, alone, batch, storage):
    kw = _kw(storage, L.LBM_COLL_REGULARIZED)
    sim = L.lbm_create(37, nx, ny, 0.8, 0.05, L.make_geometry(**kw))
    try:
        assert L.lbm_info(sim)["variant"] == alone
    finally:
        L.lbm_destroy(sim)
    b = L.lbm_batch_create(37, storage, L.LBM_COLL_REGULARIZED)
    try:
        inst = L.lbm_batch_instance(b, L.lbm_batch_add(b, L.make_instance(37, nx, ny, 0.8, 0.05, 4, **kw)))
        assert L.lbm_info(inst)["variant"] == batch
    finally:
        L.lbm_batch_destroy(b)


@pytest.mark.parametrize("nx,ny,variant", [(200, 200, 2), (200, 201, 31), (96, 900, 2), (256, 256, 31)])
def test_pairs_on_small_grids_with_boundary_nodes(nx, ny, variant):
    kw = dict(_kw(L.LBM_STORE_F16, L.LBM_COLL_REGULARIZED), kind=L.LBM_GEOM_PLATE)
    sim = L.lbm_create(37, nx, ny, 0.8, 0.05, L.make_geometry(**kw))
    try:
        assert L.lbm_info(sim)["variant"] == variant
    finally:
        L.lbm_destroy(sim)


def test_plain_bgk_keeps_one_node_per_thread():
    sim = L.lbm_create(37, 1024, 1024, 0.8, 0.05, L.make_geometry(**_kw(L.LBM_STORE_F16, L.LBM_COLL_BGK)))
    try:
        assert L.lbm_info(sim)["variant"] == 2
    finally:
        L.lbm_destroy(sim)


@pytest.mark.parametrize("storage,nx,ny,alone,batch", [
    (L.LBM_STORE_F32, 32, 9000, 0, 0), (L.LBM_STORE_F32, 33, 9000, 30, 30), (L.LBM_STORE_F32, 512, 512, 0, 30),
    (L.LBM_STORE_F32, 512, 513, 30, 30), (L.LBM_STORE_F16, 24, 9000, 0, 0), (L.LBM_STORE_F16, 256, 512, 0, 30),
    (L.LBM_STORE_F16, 256, 513, 30, 30), (L.LBM_STORE_F64, 1024, 512, 0, 0)])
def test_d2q9(storage, nx, ny, alone, batch):
    kw = dict(kind=L.LBM_GEOM_NONE, u0=1e-3, storage=storage)
    sim = L.lbm_create(9, nx, ny, 0.8, 0.05, L.make_geometry(**kw))
    b = L.lbm_batch_create(9, storage, L.LBM_COLL_REGULARIZED)
    try:
        assert L.lbm_info(sim)["variant"] == alone
        inst = L.lbm_batch_instance(b, L.lbm_batch_add(b, L.make_instance(9, nx, ny, 0.8, 0.05, 4, **kw)))
        assert L.lbm_info(inst)["variant"] == batch
    finally:
        L.lbm_batch_destroy(b)
        L.lbm_destroy(sim)
