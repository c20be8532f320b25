"""Arcs counted in stats mode by the tuned multi-source SSSP: the flagged
vertices' arcs of every round, in both forms of a round."""
import numpy as np
import pytest

from paper_2012_07990_gb300 import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 9, 32])
@pytest.mark.parametrize("isolated", [0, 5000])
def test_arcs_of_a_star(k, isolated):
    """A hub and 40 leaves with equal weights, all sources at the hub: the hub's
    arcs, then one arc of every leaf, then nothing.  With the isolated vertices
    the frontiers are small enough for lists, without them every round sweeps."""
    from paper_2012_07990_gb300 import g2
    u = np.zeros(40, int)
    g = gg.from_arcs(41 + isolated, u, np.arange(1, 41))
    dg = g2.load_graph(g, np.ones(g.m, np.int32))
    dist = torch.empty((k, g.n), dtype=torch.int32, device="cuda")
    g2.g2_set_count_arcs(True)
    try:
        g2.g2_sssp_batch(dg, np.zeros(k, np.int32), 64, dist)
        stats = g2.g2_last_stats()
    finally:
        g2.g2_set_count_arcs(False)
    assert stats["iterations"] == 2 and stats["arcs_examined"] == 80
