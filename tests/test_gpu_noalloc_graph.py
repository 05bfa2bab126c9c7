"""lbm_step_noalloc calls share one scratch array.  Every call that does not overlap another one must give its
own force, whatever ran before it: calls recorded into a graph and replayed between ordinary ones, long rows
of ordinary calls, and calls that follow others which did overlap (and whose own forces are unspecified)."""
import pytest

from paper_0904_4504_gb300 import lbm as L

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

# a plate whose body links fill several force groups, and one whose links fit in one
PLATES = {"groups": (37, 400, 24), "one-group": (9, 16, 12)}


class _Caller:
    """A simulation, two population buffers of a caller and the forces that lbm_step gives from rest."""

    def __init__(self, Q, nx, ny, wall=L.LBM_SCHEME_BOUNCEBACK):
        self.geom = L.make_geometry(kind=L.LBM_GEOM_PLATE, drive=L.LBM_DRIVE_WALL, u0=2e-3, eq_order=4 if Q == 37 else 2,
                                    storage=L.LBM_STORE_F64, wall_scheme=wall)
        self.sim = L.lbm_create(Q, nx, ny, 0.8, 0.05, self.geom)
        self.buf = [torch.zeros(Q * ny * L.lbm_info(self.sim)["pitch"], dtype=torch.float64, device="cuda") for _ in (0, 1)]
        own = L.lbm_create(Q, nx, ny, 0.8, 0.05, self.geom)
        L.lbm_step(own, 2)
        self.want = torch.from_numpy(L.lbm_force_history(own))
        L.lbm_destroy(own)
        self.force = torch.zeros((2, 2), dtype=torch.float64, device="cuda")
        self.zero = torch.zeros_like(self.buf[0])

    def two_steps(self, stream=None):
        """From rest: the forces of steps 0 and 1."""
        self.buf[0].copy_(self.zero)
        a, b = (t.data_ptr() for t in self.buf)
        L.lbm_step_noalloc(self.sim, 0, a, b, self.force[0].data_ptr(), stream or torch.cuda.current_stream())
        L.lbm_step_noalloc(self.sim, 1, b, a, self.force[1].data_ptr(), stream or torch.cuda.current_stream())

    def right(self):
        torch.cuda.synchronize()
        ok = torch.equal(self.force.cpu(), self.want)
        self.force.fill_(float("nan"))
        return ok

    def record(self):
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            self.two_steps(stream)
        return graph

    def close(self):
        torch.cuda.synchronize()
        L.lbm_destroy(self.sim)


@pytest.mark.parametrize("wall", [L.LBM_SCHEME_BOUNCEBACK, L.LBM_SCHEME_DIFFUSE], ids=["bounce", "diffuse"])
@pytest.mark.parametrize("shape", PLATES.values(), ids=list(PLATES))
def test_recorded_and_ordinary_calls(shape, wall):
    c = _Caller(*shape, wall)
    try:
        c.two_steps()
        assert c.right()
        graph = c.record()
        for k in range(100):
            graph.replay()
            assert c.right(), k
            if k % 3 == 0:
                c.two_steps()
                assert c.right(), k
        for k in range(1300):  # and without waiting between them, past each half of the tickets
            c.two_steps()
            if k % 50 == 7:
                graph.replay()
        assert c.right()
    finally:
        c.close()


def test_calls_after_overlapping_ones():
    """Two callers' rows of calls on two streams at once, then each by itself."""
    one, two = _Caller(37, 400, 24), _Caller(37, 1500, 24)
    try:
        one.two_steps()
        assert one.right()
        graph = one.record()
        for _ in range(5):
            s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
            torch.cuda.synchronize()
            for _ in range(40):
                with torch.cuda.stream(s1):
                    graph.replay()
                with torch.cuda.stream(s2):
                    two.two_steps()
            torch.cuda.synchronize()
            for c in (one, two):
                c.force.fill_(float("nan"))
                c.two_steps()
                assert c.right()
            graph.replay()
            assert one.right()
    finally:
        one.close()
        two.close()
