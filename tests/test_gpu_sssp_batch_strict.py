"""STRICT multi-source SSSP at the edges of a warp's share (128 arcs): one-arc
owners, owners longer than a share, vertices without arcs between them, a last
share of 1 to 127 arcs; directed, with weights of their own on every arc."""
import numpy as np
import pytest

import oracle
from paper_2012_07990_gb300 import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _fan(sizes):
    """Vertex 0 to hubs of the given out-degrees (0: a sink), their leaves on to
    the next hub."""
    hubs = np.arange(1, len(sizes) + 1)
    u, v, n = [np.zeros(len(sizes), int)], [hubs], len(sizes) + 1
    for i, k in enumerate(sizes):
        at = np.arange(n, n + k)
        u += [np.full(k, hubs[i]), at]
        v += [at, np.full(k, hubs[(i + 1) % len(sizes)])]
        n += k
    return gg.from_arcs(n, np.concatenate(u), np.concatenate(v), symmetric=False)


GRAPHS = {
    "shares": lambda: _fan([1, 127, 128, 129, 0, 255, 256, 257, 0, 0, 1000, 3]),
    "one_arc": lambda: gg.from_arcs(600, np.arange(599), np.arange(1, 600), symmetric=False),
    "one_share": lambda: gg.star(129),
    "rmat": lambda: gg.rmat(11, seed=4),
}


@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("k", [1, 5, 32])
@pytest.mark.parametrize("delta", [0, 64])
def test_strict(name, k, delta):
    from paper_2012_07990_gb300 import g2
    g = GRAPHS[name]()
    w = np.random.default_rng(3).integers(1, 256, g.m).astype(np.int32)
    srcs = np.random.default_rng(k).integers(0, g.n, k).astype(np.int32)
    srcs[0] = 0
    dg = g2.load_graph(g, w)
    dist = torch.full((k, g.n), -7, dtype=torch.int32, device="cuda")
    g2.g2_sssp_batch(dg, srcs, delta, dist, g2.schedule("STRICT"))
    got = dist.cpu().numpy()
    for i, s in enumerate(srcs):
        assert np.array_equal(got[i], oracle.sssp(g.n, g.rowptr, g.col, w, int(s))), i
