"""Multi-source BFS where its rounds change form, bit-exact against the oracle:
lists at the edges of a thread's, a warp's and a piece's share (32, 2,048
arcs), more levels than the bit planes hold (31), sources in components that
end early, directed graphs, and every PUSH load balancing beside PULL rounds
(they share the handle's workspace)."""
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


def _hubs_and_tail(tail, symmetric=True):
    """Hubs of 31 .. 5,000 leaves in a chain, leaves shared between neighbours,
    a tail path behind the last, a pair and an isolated vertex apart."""
    u, v, n, prev = [], [], 0, None
    for k in (31, 32, 33, 36, 161, 2047, 2048, 2049, 5000):
        leaves = np.arange(n + 1, n + 1 + k)
        u.append(np.full(k, n))
        v.append(leaves)
        if prev is not None:
            u += [np.array([prev]), leaves[::2]]
            v += [np.array([n]), np.full(leaves[::2].size, prev)]
        prev, n = n, n + 1 + k
    path = np.concatenate([[prev], np.arange(n, n + tail)])
    u += [path[:-1], np.array([n + tail])]
    v += [path[1:], np.array([n + tail + 1])]
    return gg.from_arcs(n + tail + 3, np.concatenate(u), np.concatenate(v), symmetric=symmetric)


GRAPHS = {
    "levels12": lambda: _hubs_and_tail(3),
    "levels40": lambda: _hubs_and_tail(33),
    "levels140": lambda: _hubs_and_tail(130),
    "directed": lambda: _hubs_and_tail(40, symmetric=False),
    "rmat12": lambda: gg.rmat(12, seed=8),
}


def _hybrids(g2):
    pull = g2.schedule("VERTEX_BASED", direction=g2.G2_PULL)
    yield None
    yield pull
    for lb in ("STRICT", "ETWC", "TWC", "WM"):
        yield g2.hybrid(g2.schedule(lb), pull, 0.01)


@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("k", [1, 33, 64])
def test_ms_bfs(g2, name, k):
    g = GRAPHS[name]()
    srcs = np.random.default_rng(k).integers(0, g.n, k).astype(np.int32)
    srcs[-1] = 0
    if k > 3:
        srcs[:3] = [g.n - 1, g.n - 2, g.n - 4]     # isolated, one of a pair, the tail's end
    want = np.stack([oracle.bfs(g.n, g.rowptr, g.col, int(s), False)[0] for s in srcs])
    dg = g2.load_graph(g)
    depth = torch.empty((k, g.n), dtype=torch.int32, device="cuda")
    for sched in _hybrids(g2):
        depth.fill_(-9)
        g2.g2_bfs_batch(dg, srcs, depth, sched)
        assert np.array_equal(depth.cpu().numpy(), want)
