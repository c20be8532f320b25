"""Delta-stepping's NULL schedule on graphs that are not of bounded degree (the
near/far loop with STRICT rounds in one launch), bit-exact against the oracle:
near lists around the size that every CTA scans itself (1,024), hubs, long
paths behind a hub, directed graphs, unreached vertices, deltas below, inside
and above the weights' range; and the refusals around it."""
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


def _two_stars(leaves):
    """Two hubs that share `leaves` leaves, a tail behind one, a pair apart."""
    l = np.arange(2, leaves + 2)
    tail = np.arange(leaves + 2, leaves + 80)
    u = np.concatenate([np.zeros(leaves, int), np.ones(leaves, int), [1], tail[:-1], [leaves + 80]])
    v = np.concatenate([l, l, [tail[0]], tail[1:], [leaves + 81]])
    return gg.from_arcs(leaves + 83, u, v)


GRAPHS = {
    **{f"stars{n}": (lambda n=n: _two_stars(n)) for n in (33, 1023, 1024, 1025, 4097)},
    "rmat13": lambda: gg.rmat(13, seed=4),
    "directed": lambda: gg.gnp(400, 0.2, 3, symmetric=False),
}


@pytest.mark.parametrize("delta", [1, 64, 300])
@pytest.mark.parametrize("name", list(GRAPHS))
def test_sssp_null(g2, name, delta):
    g = GRAPHS[name]()
    w = gg.pair_weights(g, 255, seed=3)
    dg = g2.load_graph(g, w)
    dist = torch.empty(g.n, dtype=torch.int32, device="cuda")
    for src in (0, g.n // 2, g.n - 1):
        g2.g2_sssp_delta(dg, src, delta, dist)
        assert np.array_equal(dist.cpu().numpy(), oracle.sssp(g.n, g.rowptr, g.col, w, src))


def test_strict_fusion_stays_refused(g2):
    g = gg.star(50)
    dg = g2.load_graph(g, gg.pair_weights(g, 9))
    dist = torch.empty(g.n, dtype=torch.int32, device="cuda")
    with pytest.raises(g2.G2Error) as e:
        g2.g2_sssp_delta(dg, 0, 4, dist, g2.schedule("STRICT", kernel_fusion=True))
    assert e.value.status == g2.G2_EUNSUPPORTED


def test_overflow_is_reported(g2):
    g = gg.star(41)
    w = np.ones(g.m, np.int32)
    u = np.repeat(np.arange(g.n), g.degrees())
    w[(u == 0) & (g.col == 40)] = 2**31 - 2
    dg = g2.load_graph(g, w)
    dist = torch.empty(g.n, dtype=torch.int32, device="cuda")
    with pytest.raises(g2.G2Error) as e:
        g2.g2_sssp_delta(dg, 1, 64, dist)
    assert e.value.status == g2.G2_EOVERFLOW
