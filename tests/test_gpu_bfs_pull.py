"""The fused hybrid's PULL levels, bit-exact against the oracle where the ends
of a warp's four bitmap words and of the vertex range fall (n around 32, 128 and
256), where the warps take a second turn (n above 152 SMs x 4 CTAs x 1,024), and
where lists of very different lengths share a lane."""
import numpy as np
import pytest

import oracle
from paper_2012_07990_gb300 import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g2():
    from paper_2012_07990_gb300 import g2 as m
    return m


def _check(g2, g, src):
    pull = g2.schedule("VERTEX_BASED", direction=g2.G2_PULL, pull_frontier=g2.G2_BITMAP,
                       frontier_creation=g2.G2_UNFUSED_BITMAP, dedup=False, kernel_fusion=True)
    want_depth, want_parent = oracle.bfs_graph(g, src)
    dg = g2.load_graph(g)
    depth = torch.empty(g.n, dtype=torch.int32, device="cuda")
    parent = torch.empty_like(depth)
    for sched in (None, g2.hybrid(g2.schedule("STRICT", kernel_fusion=True), pull, 0.0)):
        g2.g2_bfs(dg, src, depth, parent, sched)
        assert np.array_equal(depth.cpu().numpy(), want_depth)
        assert np.array_equal(parent.cpu().numpy(), want_parent)


@pytest.mark.parametrize("n", [33, 127, 128, 129, 255, 257, 1001])
@pytest.mark.parametrize("symmetric", [True, False])
def test_pull_ends(g2, n, symmetric):
    r = np.random.default_rng(n)
    hub = np.zeros(n - 1, dtype=np.int64)
    u, v = r.integers(0, n, 2 * n), r.integers(0, n, 2 * n)
    g = gg.from_arcs(n, np.concatenate([hub[: n // 3], u]), np.concatenate([np.arange(1, n)[: n // 3], v]),
                     symmetric=symmetric)
    _check(g2, g, int(g.col[0]))


def test_pull_second_turn(g2):
    n = 152 * 4 * 1024 + 77
    r = np.random.default_rng(3)
    hub = r.permutation(n)[: n // 2]
    tail = np.arange(n - 200, n)
    g = gg.from_arcs(n, np.concatenate([np.full(hub.size, 5), tail[:-1]]), np.concatenate([hub, tail[1:]]))
    _check(g2, g, 5)


def _hub_levels(first, hubs, leaves, n, symmetric):
    """Vertex 0 -> `first` vertices; the last of them -> `hubs` vertices of
    `leaves` random neighbours each (`first` = 0: vertex 0 -> the hubs)."""
    r = np.random.default_rng(hubs + first)
    h = np.arange(1 + first, 1 + first + hubs)
    u = np.concatenate([np.zeros(first, int), np.full(hubs, first), np.repeat(h, leaves)])
    v = np.concatenate([np.arange(1, 1 + first), h, r.integers(1 + first + hubs, n, hubs * leaves)])
    return gg.from_arcs(n, u, v, symmetric=symmetric)


@pytest.mark.parametrize("symmetric", [True, False])
@pytest.mark.parametrize("first,hubs,leaves", [
    (0, 4, 150000),       # a list that every CTA scans itself
    (0, 1500, 400),       # one scanned over the grid
    (6000, 4, 150000),    # a bitmap made a list first (6,000 vertices: 3% of n)
    (6000, 1500, 400),
])
def test_few_vertices_many_arcs(g2, first, hubs, leaves, symmetric):
    """Levels of less than 2% of the vertices with more than 2^18 arcs: pulled
    by the NULL schedule, pushed by the hybrid that asks for it."""
    g = _hub_levels(first, hubs, leaves, 200_000, symmetric)
    want_depth, want_parent = oracle.bfs_graph(g, 0)
    dg = g2.load_graph(g)
    depth = torch.empty(g.n, dtype=torch.int32, device="cuda")
    parent = torch.empty_like(depth)
    pull = g2.schedule("VERTEX_BASED", direction=g2.G2_PULL, pull_frontier=g2.G2_BITMAP,
                       frontier_creation=g2.G2_UNFUSED_BITMAP, dedup=False, kernel_fusion=True)
    pulls = []
    for sched in (None, g2.hybrid(g2.schedule("STRICT", kernel_fusion=True), pull, 0.02)):
        g2.g2_bfs(dg, 0, depth, parent, sched)
        assert np.array_equal(depth.cpu().numpy(), want_depth)
        assert np.array_equal(parent.cpu().numpy(), want_parent)
        pulls.append(g2.g2_last_stats()["pull_rounds"])
    assert pulls[0] == pulls[1] + 1
