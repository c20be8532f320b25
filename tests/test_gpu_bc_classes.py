"""Betweenness centrality where its level passes change granularity, against the
long double oracle: degrees at the edges of the classes (8 / 9, 128 / 129,
2,048 and pieces of 2,048 arcs), more levels than the counting sort keeps in
shared memory (64), directed graphs (in- and out-degrees grouped apart), one
source (a round per level) and several (depths in one launch)."""
import numpy as np
import pytest

import oracle
from paper_2012_07990_gb300 import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BC_REL, BC_ABS = 1e-6, 1e-12


@pytest.fixture(scope="module")
def g2():
    from paper_2012_07990_gb300 import g2 as m
    return m


def _hub_tree(symmetric=True):
    """A root joined to hubs of 7 .. 6,200 leaves, every leaf of a hub also to
    the next hub (many shortest paths), and a tail of 150 vertices."""
    u, v, n, prev = [], [], 1, 0
    for k in (7, 8, 9, 126, 127, 128, 2046, 2047, 2048, 4096, 6200):
        hub, leaves = n, np.arange(n + 1, n + 1 + k)
        u += [np.array([0]), np.full(k, hub), leaves[::3]]
        v += [np.array([hub]), leaves, np.full(leaves[::3].size, prev)]
        prev, n = hub, n + 1 + k
    tail = np.arange(n, n + 150)
    u += [np.array([prev]), tail[:-1]]
    v += [np.array([tail[0]]), tail[1:]]
    u, v = np.concatenate(u), np.concatenate(v)
    return gg.from_arcs(n + 150, u, v, symmetric=symmetric), tail[-1]


@pytest.mark.parametrize("symmetric", [True, False])
@pytest.mark.parametrize("k", [1, 4])
def test_bc_classes(g2, symmetric, k):
    g, end = _hub_tree(symmetric)
    srcs = np.array([end if symmetric else 0, 0, 5, 300], np.int32)[:k]
    want = oracle.bc_graph(g, srcs)
    bc = torch.empty(g.n, dtype=torch.float64, device="cuda")
    dg = g2.load_graph(g)
    for sched in (None, g2.schedule("WM")):
        bc.fill_(-1.0)
        g2.g2_bc(dg, srcs, bc, sched)
        got = bc.cpu().numpy()
        assert np.all(np.abs(got - want) <= BC_REL * np.abs(want) + BC_ABS * np.abs(want).max())
