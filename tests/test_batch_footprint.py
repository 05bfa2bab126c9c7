"""lbm_batch_footprint bounds what an instance's lists make it hold: 24 bytes a boundary node, 8 a body link (bounce-
back), the link masks by node, the populations and the history.  Host only."""
import numpy as np
import pytest

from paper_0904_4504_gb300 import builder as B
from paper_0904_4504_gb300 import lbm as L


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def porous(nx, ny, seed=2):
    """Single body nodes (an eighth of the grid) and some wall ones."""
    rng = np.random.default_rng(seed)
    return rng.choice(np.array([0, 1, 2], np.uint8), (ny, nx), p=[0.85, 0.125, 0.025])


GEOMETRY = {
    "beam": lambda nx, ny: dict(kind=L.LBM_GEOM_BEAM, lx=nx // 3, ly=ny // 4),
    "thin": lambda nx, ny: dict(kind=L.LBM_GEOM_BEAM, lx=nx - 6, ly=1),
    "dot": lambda nx, ny: dict(kind=L.LBM_GEOM_BEAM, lx=1, ly=2),
    "plate": lambda nx, ny: dict(kind=L.LBM_GEOM_PLATE),
    "porous": lambda nx, ny: dict(kind=L.LBM_GEOM_MASK, mask=porous(nx, ny)),
    "open": lambda nx, ny: dict(kind=L.LBM_GEOM_NONE),
}


@pytest.mark.parametrize("wall", [L.LBM_SCHEME_BOUNCEBACK, L.LBM_SCHEME_DIFFUSE], ids=["bounce", "diffuse"])
@pytest.mark.parametrize("geometry", GEOMETRY)
@pytest.mark.parametrize("Q,nx,ny", [(37, 200, 200), (37, 2048, 8), (37, 45, 300), (9, 4096, 5), (9, 61, 64)])
def test_footprint_covers_the_lists(Q, nx, ny, geometry, wall):
    kw = GEOMETRY[geometry](nx, ny)
    cls, body, wall_links, n_fluid, nb = L.lbm_geometry_links(Q, nx, ny, L.make_geometry(**kw))
    nfl = int(np.bitwise_count(body).sum()) if wall == L.LBM_SCHEME_BOUNCEBACK else 0
    for es, storage in ((8, L.LBM_STORE_F64), (2, L.LBM_STORE_F16)):
        pitch = -(-nx * es // 128) * 128 // es
        steps = 300
        by_node = 17 if wall == L.LBM_SCHEME_BOUNCEBACK else 1   # classes; link masks, which tile kernels read
        holds = (2 * Q * es + by_node) * ny * pitch + 24 * nb + 8 * nfl + 16 * 1024 + 128 * steps
        d = L.make_instance(Q, nx, ny, 0.8, 0.05, steps, storage=storage, wall_scheme=wall, u0=1e-3, **kw)
        assert L.lbm_batch_footprint(d) >= holds, (storage, nb, nfl)


def test_footprint_of_what_cannot_be_added():
    """Sizes and geometries that lbm_batch_add refuses still have the footprint of their sizes."""
    same = L.lbm_batch_footprint(L.make_instance(37, 64, 48, 0.8, 0.05, 10, kind=L.LBM_GEOM_NONE))
    for kw in (dict(kind=L.LBM_GEOM_MASK), dict(kind=L.LBM_GEOM_BEAM, lx=64, ly=3), dict(kind=9)):
        assert L.lbm_batch_footprint(L.make_instance(37, 64, 48, 0.8, 0.05, 10, **kw)) == same
    for nx, ny in ((1, 1), (3, 900), (1 << 20, 1 << 12)):
        assert L.lbm_batch_footprint(L.make_instance(37, nx, ny, 0.8, 0.05, 10, kind=L.LBM_GEOM_PLATE)) > 2 * 37 * 4 * nx * ny
