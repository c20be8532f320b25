"""One PUSH round of RELAX_MIN / LABEL_MIN against numpy, bit-exact: sources
act with their values from before the round, whatever the load balancing.

The graphs and frontiers sit at the edges of the load balancers' shares: list
lengths around a warp, a CTA and a hand-off piece (32, 256, 1,024 arcs), runs
of vertices without arcs longer than a STRICT tile, one-arc owners, a frontier
that repeats a hub past the room of ETWC's hand-off list."""
import numpy as np
import pytest

from paper_2012_07990_gb300 import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

INF = 2**31 - 1


@pytest.fixture(scope="module")
def g2():
    from paper_2012_07990_gb300 import g2 as m
    return m


def _edges_of_shares():
    """Stars of 31 .. 4,097 leaves, then 3,000 isolated vertices."""
    u, v, n = [], [], 0
    for k in (1, 31, 32, 33, 255, 256, 257, 1023, 1024, 1025, 1281, 4097):
        u.append(np.full(k, n))
        v.append(np.arange(n + 1, n + 1 + k))
        n += k + 1
    return gg.from_arcs(n + 3000, np.concatenate(u), np.concatenate(v))


def _cases():
    shares = _edges_of_shares()
    hubs = np.nonzero(shares.degrees() > 1)[0]
    leaves = np.nonzero(shares.degrees() == 1)[0]
    empty = np.nonzero(shares.degrees() == 0)[0]
    rmat = gg.rmat(13, seed=2)
    rng = np.random.default_rng(4)
    star = gg.star(5000)
    return {
        "hubs": (shares, hubs),
        "leaves": (shares, leaves),                                    # one arc each
        "empty_between": (shares, np.concatenate([hubs[:5], empty, hubs[5:], empty[:1500], leaves[:40]])),
        "rmat_sorted": (rmat, np.sort(rng.choice(rmat.n, 2500, replace=False))),
        "rmat_one": (rmat, np.array([0])),
        "rmat_all": (rmat, np.arange(rmat.n)),
        "repeated_hub": (star, np.concatenate([np.zeros(1000, int), [7, 9]])),
    }


CASES = _cases()


@pytest.mark.parametrize("lb", ["VERTEX_BASED", "WM", "CM", "STRICT", "ETWC", "TWC"])
@pytest.mark.parametrize("name", list(CASES))
def test_push_round(g2, name, lb):
    g, verts = CASES[name]
    w = gg.pair_weights(g, 50, seed=1)
    dg = g2.load_graph(g, w)
    rng = np.random.default_rng(1)
    d0 = rng.integers(0, 300, g.n).astype(np.int32)
    d0[rng.random(g.n) < 0.3] = INF
    src = np.repeat(np.arange(g.n), g.degrees())
    on = np.isin(src, verts)
    fin, fout = (g2.g2_frontier_create(dg, g2.G2_FRONTIER_SPARSE) for _ in range(2))
    fin.set(verts)
    for op, step in ((g2.G2_OP_RELAX_MIN, w), (g2.G2_OP_LABEL_MIN, np.zeros(g.m, np.int32))):
        reach = on & (d0[src] != INF) if op == g2.G2_OP_RELAX_MIN else on
        want = d0.copy()
        np.minimum.at(want, g.col[reach], d0[src[reach]] + step[reach])
        val = torch.from_numpy(d0).cuda()
        size = g2.g2_edgeset_apply(dg, op, fin, val, None, g2.schedule(lb), fout)
        assert np.array_equal(val.cpu().numpy(), want)
        lst = torch.empty(g.n, dtype=torch.int32, device="cuda")
        assert fout.to_list(lst) == size == int((want < d0).sum())
        assert np.array_equal(np.sort(lst[:size].cpu().numpy()), np.nonzero(want < d0)[0])
