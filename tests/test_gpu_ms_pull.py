"""Multi-source BFS PULL rounds about the lines between their forms, bit-exact
against the oracle: lists that a thread walks whole (up to 128 arcs, where none
is longer), lists left to a warp, several such lists per warp, and sources few
enough for direct depths (16) or not, in searches of few and of many levels."""
import numpy as np
import pytest

import oracle
from paper_2012_07990_gb300 import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(g, k, seed=0):
    from paper_2012_07990_gb300 import g2
    srcs = np.random.default_rng(seed + k).integers(0, g.n, k).astype(np.int32)
    srcs[-1] = 0
    want = np.stack([oracle.bfs(g.n, g.rowptr, g.col, int(s), False)[0] for s in srcs])
    dg = g2.load_graph(g)
    depth = torch.empty((k, g.n), dtype=torch.int32, device="cuda")
    pull = g2.schedule("VERTEX_BASED", direction=g2.G2_PULL)
    for sched in (None, pull, g2.hybrid(g2.schedule("STRICT"), pull, 0.02)):
        depth.fill_(-9)
        g2.g2_bfs_batch(dg, srcs, depth, sched)
        assert np.array_equal(depth.cpu().numpy(), want)


def _ring(degrees, tail):
    """Hubs of the given degrees around a ring of shared leaves, and a tail."""
    u, v, n = [], [], len(degrees)
    leaves = n + np.arange(max(degrees) + 7)
    for i, d in enumerate(degrees):
        u.append(np.full(d, i))
        v.append(leaves[(np.arange(d) + 3 * i) % leaves.size])
    n += leaves.size
    path = np.concatenate([[leaves[0]], np.arange(n, n + tail)])
    return gg.from_arcs(n + tail + 2, np.concatenate(u + [path[:-1]]), np.concatenate(v + [path[1:]]))


@pytest.mark.parametrize("k", [1, 16, 17, 64])
@pytest.mark.parametrize("top", [31, 32, 33, 127, 128, 129, 2047, 2048])
@pytest.mark.parametrize("tail", [2, 45])
def test_longest_list(k, top, tail):
    _check(_ring([1, 4, 5, min(top, 36), min(top, 64), top], tail), k)


@pytest.mark.parametrize("k", [5, 20, 64])
@pytest.mark.parametrize("symmetric", [True, False])
def test_many_lists_per_warp(k, symmetric):
    """40,000 vertices of some 44 arcs in a band, and one of 300."""
    r = np.random.default_rng(1)
    i = np.repeat(np.arange(40000), 22 if symmetric else 44)
    j = i + r.integers(1, 3000, i.size)
    u = np.concatenate([i[j < 40000], np.full(300, 20000)])
    v = np.concatenate([j[j < 40000], r.integers(0, 40000, 300)])
    _check(gg.from_arcs(40000, u[u != v], v[u != v], symmetric=symmetric), k)
