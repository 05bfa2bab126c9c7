"""The library's work is ordered on its own streams: work that the caller has queued on the default stream
(here: some 50 ms of it, put there just before each call) changes no result."""
import numpy as np
import pytest

from paper_0904_4504_gb300 import lbm as L

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


def _busy(on):
    if on:
        torch.cuda._sleep(100_000_000)


def _geom(layout):
    return L.make_geometry(kind=L.LBM_GEOM_BEAM, lx=13, ly=11, drive=L.LBM_DRIVE_WALL, u0=2e-3, eq_order=4, layout=layout)


@pytest.mark.parametrize("layout", [L.LBM_LAYOUT_AB, L.LBM_LAYOUT_AA], ids=["two", "inplace"])
@pytest.mark.parametrize("calls", [(1500,), (900, 500, 2500)], ids=["first", "again"])
def test_history_that_grows(layout, calls):
    """The history holds 1024 steps at first: the calls make it grow once or twice."""
    got = []
    for busy in (False, True):
        sim = L.lbm_create(37, 61, 47, 0.8, 0.05, _geom(layout))
        try:
            for n in calls:
                _busy(busy)
                L.lbm_step(sim, n)
            got.append(L.lbm_force_history(sim))
        finally:
            torch.cuda.synchronize()
            L.lbm_destroy(sim)
    assert got[0].shape == (sum(calls), 2) and (np.abs(got[0]).max(1) > 0).all()
    assert (got[0] == got[1]).all()


def test_persistent_batch():
    """Counters and step tables of a batch that is created, filled and run behind queued work."""
    got = []
    for busy in (False, True):
        torch.cuda.synchronize()
        _busy(busy)
        batch = L.lbm_batch_create(37, L.LBM_STORE_F32, L.LBM_COLL_REGULARIZED)
        try:
            L.lbm_batch_set_mode(batch, L.LBM_BATCH_PERSISTENT)
            slots = [L.lbm_batch_add(batch, L.make_instance(37, n, 41, 0.8, 0.05, 1100, kind=L.LBM_GEOM_BEAM, lx=7, ly=9,
                                                            drive=L.LBM_DRIVE_WALL, u0=2e-3, eq_order=4)) for n in (45, 70)]
            _busy(busy)
            L.lbm_batch_run(batch, 1100)
            L.lbm_batch_synchronize(batch)
            got.append([L.lbm_force_history(L.lbm_batch_instance(batch, s)) for s in slots])
        finally:
            torch.cuda.synchronize()
            L.lbm_batch_destroy(batch)
    for idle, queued in zip(*got):
        assert (np.abs(idle).max(1) > 0).all() and (idle == queued).all()


def test_set_state():
    rng = np.random.default_rng(3)
    got = []
    g = rng.uniform(-1e-4, 1e-4, (37, 47, 61))
    for busy in (False, True):
        sim = L.lbm_create(37, 61, 47, 0.8, 0.05, _geom(L.LBM_LAYOUT_AB))
        try:
            _busy(busy)
            L.lbm_set_state(sim, g)
            _busy(busy)
            L.lbm_step(sim, 4)
            got.append((L.lbm_get_state(sim), L.lbm_force_history(sim)))
        finally:
            torch.cuda.synchronize()
            L.lbm_destroy(sim)
    assert (got[0][0] == got[1][0]).all() and (got[0][1] == got[1][1]).all()
