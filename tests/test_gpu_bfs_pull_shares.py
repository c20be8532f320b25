"""The fused hybrid's PULL levels about the line between one and four bitmap
words a warp (1,216 words with one CTA per SM on 152 SMs), where four fill
every warp (4,864), and on a band whose levels leave most lists without a hit;
bit-exact against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2012_07990_gb300 import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LINE = 152 * 8 * 32


def _check(g, src):
    from paper_2012_07990_gb300 import g2
    pull = g2.schedule("VERTEX_BASED", direction=g2.G2_PULL, pull_frontier=g2.G2_BITMAP,
                       frontier_creation=g2.G2_UNFUSED_BITMAP, dedup=False, kernel_fusion=True)
    want_depth, want_parent = oracle.bfs_graph(g, src)
    dg = g2.load_graph(g)
    depth = torch.empty(g.n, dtype=torch.int32, device="cuda")
    parent = torch.empty_like(depth)
    for lb in ("STRICT", "WM"):
        g2.g2_bfs(dg, src, depth, parent, g2.hybrid(g2.schedule(lb, kernel_fusion=True), pull, 0.0))
        assert np.array_equal(depth.cpu().numpy(), want_depth)
        assert np.array_equal(parent.cpu().numpy(), want_parent)
    g2.g2_bfs(dg, src, depth, parent)
    assert np.array_equal(depth.cpu().numpy(), want_depth)
    assert np.array_equal(parent.cpu().numpy(), want_parent)


@pytest.mark.parametrize("n", [line + d for line in (LINE, 4 * LINE) for d in (-64, -31, 0, 1, 97)])
def test_about_the_line(monkeypatch, n):
    monkeypatch.setenv("G2_FUSED_DO_CTAS_PER_SM", "1")
    r = np.random.default_rng(n)
    hub = r.permutation(n)[: n // 2]
    tail = np.arange(n - 100, n)
    _check(gg.from_arcs(n, np.concatenate([np.full(hub.size, 5), tail[:-1]]), np.concatenate([hub, tail[1:]])), 5)


@pytest.mark.parametrize("symmetric", [True, False])
def test_band(symmetric):
    r = np.random.default_rng(2)
    i = np.repeat(np.arange(20000), 24)
    j = i + r.integers(1, 700, i.size)
    _check(gg.from_arcs(20000, i[j < 20000], j[j < 20000], symmetric=symmetric), 3)
