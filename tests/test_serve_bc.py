"""BC batches of the query server: with several slots a batch on a power-law
graph runs by rounds (no cooperative launch beside the other slots), with one
slot by the library's schedule."""
import pytest

from paper_2012_07990_gb300 import graphgen as gg
from paper_2012_07990_gb300 import serve

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


class Spy:
    """The binding, with the schedules that g2_bc is given kept."""

    def __init__(self, g2):
        self._g2, self.scheds = g2, []

    def __getattr__(self, name):
        return getattr(self._g2, name)

    def g2_bc(self, view, srcs, out, sched):
        self.scheds.append(sched)
        self._g2.g2_bc(view, srcs, out, sched)


@pytest.mark.parametrize("k", [1, 3])
@pytest.mark.parametrize("slots", [1, 4])
def test_schedule_of_bc_batches(k, slots):
    from paper_2012_07990_gb300 import g2
    specs = [serve.GraphSpec("rmat10", lambda: gg.rmat(10, seed=1), 255, 64),
             serve.GraphSpec("grid40", lambda: gg.road_grid(40, seed=1), 1000, 4096, True)]
    pool = serve.GraphPool(g2, specs)
    spy = Spy(g2)
    ex = serve.GpuExecutor(spy, pool, slots=slots)
    for graph in ("rmat10", "grid40"):
        ex.execute(slots - 1, [serve.Request(i, 0.0, graph, "bc", 7 + i) for i in range(k)])
    rounds = slots > 1 and k > 1
    assert spy.scheds == [ex.powerlaw_bfs if rounds else None, ex.fused]
    assert not rounds or ex.powerlaw_bfs.s1.kernel_fusion == 0
