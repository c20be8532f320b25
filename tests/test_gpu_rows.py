"""Multi-source SSSP over distance rows (the NULL schedule of g2_sssp_batch on
symmetric graphs that are not of bounded degree), bit-exact against the oracle:
every row width (8, 16, 32) and its edges, runs of a vertex's in-arcs across a
warp's share (a hub), rounds of both directions (a long path behind a hub), a
ragged last share, isolated sources, repeated sources, and the overflow rule."""
import numpy as np
import pytest

import oracle
from paper_2012_07990_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g2():
    from paper_2012_07990_gb300 import g2 as m
    return m


def _lollipop(leaves, tail):
    """A hub with `leaves` leaves and a path of `tail` vertices."""
    star = np.stack([np.zeros(leaves, int), np.arange(1, leaves + 1)])
    path = np.stack([np.arange(leaves, leaves + tail - 1), np.arange(leaves + 1, leaves + tail)])
    u, v = np.concatenate([star, path], axis=1)
    return gg.from_arcs(leaves + tail + 3, u, v)   # three isolated vertices at the end


GRAPHS = {
    "rmat12": lambda: gg.rmat(12, seed=3),
    "gnp": lambda: gg.gnp(301, 0.3, 5),
    "lollipop": lambda: _lollipop(1000, 4000),
    "hubs": lambda: gg.complete(70),
}


@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("k", [1, 8, 9, 16, 17, 32])
def test_rows(g2, name, k):
    import torch
    g = GRAPHS[name]()
    w = gg.pair_weights(g, 255, seed=2)
    srcs = np.random.default_rng(k).integers(0, g.n, k).astype(np.int32)
    if k > 1:
        srcs[-1], srcs[0] = srcs[0], g.n - 1
    dg = g2.load_graph(g, w)
    dist = torch.full((k, g.n), -7, dtype=torch.int32, device="cuda")
    for delta in (0, 64):
        dist.fill_(-7)
        g2.g2_sssp_batch(dg, srcs, delta, dist)
        got = dist.cpu().numpy()
        for i in range(k):
            assert np.array_equal(got[i], oracle.sssp(g.n, g.rowptr, g.col, w, int(srcs[i]))), (i, delta)


@pytest.mark.parametrize("last, over", [(2**31 - 4, False), (2**31 - 3, True)])
def test_rows_overflow(g2, last, over):
    """A hub with 40 leaves, unit arcs but 0 -> 40 of weight `last`: from leaf 1
    vertex 40 lies at last + 1, and its arc back leads to last + 2, which may
    not reach INT32_MAX; the same answer as with an explicit schedule."""
    import torch
    g = gg.star(41)
    u = np.repeat(np.arange(g.n), g.degrees())
    w = np.ones(g.m, np.int32)
    w[(u == 0) & (g.col == 40)] = last
    dg = g2.load_graph(g, w)
    dist = torch.empty((1, g.n), dtype=torch.int32, device="cuda")
    for sched in (None, g2.schedule("STRICT")):
        if over:
            with pytest.raises(g2.G2Error) as e:
                g2.g2_sssp_batch(dg, [1], 64, dist, sched)
            assert e.value.status == g2.G2_EOVERFLOW
        else:
            g2.g2_sssp_batch(dg, [1], 64, dist, sched)
            want = np.full(41, 2)
            want[[0, 1, 40]] = [1, 0, last + 1]
            assert np.array_equal(dist.cpu().numpy()[0], want)
