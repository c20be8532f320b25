"""Betweenness centrality by rounds on symmetric graphs whose lists all hold at
most 32 arcs (a thread per vertex over the levels as found), against the long
double oracle; one with 33 takes the grouped form."""
import numpy as np
import pytest

import oracle
from paper_2012_07990_gb300 import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BC_REL, BC_ABS = 1e-6, 1e-12


def _graph(top):
    """Hubs of 8, 9, 31 and `top` leaves in a row, leaves shared between
    neighbours, a tail, and vertices that no source reaches."""
    u, v, n, prev = [], [], 0, None
    for k in (8, 9, 31, top):
        at = np.arange(n + 1, n + 1 + k - (prev is not None))
        u.append(np.full(at.size, n))
        v.append(at)
        if prev is not None:
            u += [np.array([prev[0]]), prev[1:4]]
            v += [np.array([n]), at[:3]]
        prev, n = np.concatenate([at[-1:], at[1:]]), n + 1 + at.size
    tail = np.arange(n, n + 70)
    u += [prev[:1], tail[:-1]]
    v += [tail[:1], tail[1:]]
    return gg.from_arcs(n + 75, np.concatenate(u), np.concatenate(v)), int(tail[-1])


@pytest.mark.parametrize("top", [32, 33])
@pytest.mark.parametrize("k", [1, 3])
@pytest.mark.parametrize("lb", ["VERTEX_BASED", "CM", "WM", "STRICT", "ETWC", "hybrid"])
def test_bc(top, k, lb):
    from paper_2012_07990_gb300 import g2
    g, end = _graph(top)
    assert g.degrees().max() == top
    srcs = np.array([end, 0, g.n - 1], np.int32)[:k]
    pull = g2.schedule("VERTEX_BASED", direction=g2.G2_PULL, pull_frontier=g2.G2_BITMAP,
                       frontier_creation=g2.G2_UNFUSED_BITMAP, dedup=False)
    sched = g2.hybrid(g2.schedule("STRICT"), pull, 0.02) if lb == "hybrid" else g2.schedule(lb)
    want = oracle.bc_graph(g, srcs)
    dg = g2.load_graph(g)
    bc = torch.empty(g.n, dtype=torch.float64, device="cuda")
    for _ in range(2):
        bc.fill_(-1.0)
        g2.g2_bc(dg, srcs, bc, sched)
        got = bc.cpu().numpy()
        assert np.all(np.abs(got - want) <= BC_REL * np.abs(want) + BC_ABS * np.abs(want).max())
