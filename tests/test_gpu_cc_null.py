"""Connected components with the NULL schedule, bit-exact against the oracle,
on graphs whose vertices' smallest neighbours are larger than themselves
(shuffled ids, hubs with the largest id), on many small components, and around
the 1,024 sampled labels."""
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


def _shuffled(g, seed):
    p = np.random.default_rng(seed).permutation(g.n)
    u = np.repeat(np.arange(g.n), g.degrees())
    return gg.from_arcs(g.n, p[u], p[g.col], symmetric=False)


def _pairs(k):
    return gg.from_arcs(2 * k + 1, np.arange(k), 2 * k - 1 - np.arange(k))


GRAPHS = {
    "one": lambda: gg.from_arcs(1, [], []),
    "isolated": lambda: gg.from_arcs(1025, [], []),
    "pairs": lambda: _pairs(700),
    "star_high": lambda: gg.from_arcs(3000, np.full(2999, 2999), np.arange(2999)),
    "path": lambda: _shuffled(gg.path(5000), 1),
    "forest": lambda: _shuffled(gg.gnp(1500, 1.1 / 1500, 2), 3),
    "union": lambda: _shuffled(gg.disjoint_union(gg.star(400), gg.cycle(700), gg.complete(30), gg.path(500)), 4),
    "rmat": lambda: _shuffled(gg.rmat(12, seed=6), 5),
    "grid": lambda: _shuffled(gg.road_grid(70, 50, seed=3), 6),
}


@pytest.mark.parametrize("name", list(GRAPHS))
def test_cc_null(g2, name):
    g = GRAPHS[name]()
    dg = g2.g2_load_csr(g.n, g.rowptr, g.col, symmetric=True)
    label = torch.empty(g.n, dtype=torch.int32, device="cuda")
    for _ in range(3):
        label.fill_(-1)
        g2.g2_cc(dg, label)
        assert np.array_equal(label.cpu().numpy(), oracle.cc(g.n, g.rowptr, g.col))
