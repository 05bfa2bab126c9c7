"""An instance of a batch holds no more device memory than the budget counts for it, and than lbm_batch_footprint says."""
import pytest

from paper_0904_4504_gb300 import lbm as L

from test_batch_footprint import GEOMETRY

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.mark.parametrize("mode", [L.LBM_BATCH_STREAMS, L.LBM_BATCH_PERSISTENT], ids=["streams", "persistent"])
@pytest.mark.parametrize("storage", [L.LBM_STORE_F32, L.LBM_STORE_F16], ids=["f32", "f16"])
@pytest.mark.parametrize("geometry", GEOMETRY)
@pytest.mark.parametrize("Q,nx,ny", [(37, 200, 200), (37, 2048, 8), (9, 4096, 5), (9, 61, 64)])
def test_an_instance_holds_no_more_than_counted(Q, nx, ny, geometry, storage, mode):
    kw = GEOMETRY[geometry](nx, ny)
    batch = L.lbm_batch_create(Q, storage, L.LBM_COLL_REGULARIZED)
    try:
        L.lbm_batch_set_mode(batch, mode)
        for steps in (4, 1500):
            d = L.make_instance(Q, nx, ny, 0.8, 0.05, steps, storage=storage, u0=1e-3, drive=L.LBM_DRIVE_WALL,
                                eq_order=4 if Q == 37 else 2, **kw)
            before = L.lbm_batch_info(batch)["used_bytes"]
            sim = L.lbm_batch_instance(batch, L.lbm_batch_add(batch, d))
            counted = L.lbm_batch_info(batch)["used_bytes"] - before
            table = 128 * steps if mode == L.LBM_BATCH_PERSISTENT else 0
            assert L.lbm_info(sim)["device_bytes"] + table <= min(counted, L.lbm_batch_footprint(d))
            if mode == L.LBM_BATCH_STREAMS:
                L.lbm_set_variant(sim, 10)  # a tile kernel: it reads the links by node
                assert L.lbm_info(sim)["device_bytes"] <= min(counted, L.lbm_batch_footprint(d))
    finally:
        L.lbm_batch_destroy(batch)


def test_a_budget_below_the_lists_is_refused():
    """A body full of holes whose sizes alone would fit the budget, and the same with the room it needs."""
    d = L.make_instance(37, 200, 200, 0.8, 0.05, 16, storage=L.LBM_STORE_F16, u0=1e-3, drive=L.LBM_DRIVE_WALL, eq_order=4,
                        **GEOMETRY["porous"](200, 200))
    sizes = L.lbm_batch_footprint(L.make_instance(37, 200, 200, 0.8, 0.05, 16, storage=L.LBM_STORE_F16, u0=1e-3))
    need = L.lbm_batch_footprint(d)
    assert need > sizes
    for budget, fits in ((sizes, False), (need, True)):
        batch = L.lbm_batch_create(37, L.LBM_STORE_F16, L.LBM_COLL_REGULARIZED, budget)
        try:
            if fits:
                L.lbm_batch_add(batch, d)
            else:
                with pytest.raises(L.LbmError) as e:
                    L.lbm_batch_add(batch, d)
                assert e.value.code == L.LBM_ENOMEM and L.lbm_batch_info(batch)["used_bytes"] == 0
        finally:
            L.lbm_batch_destroy(batch)
