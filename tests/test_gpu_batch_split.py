"""Batched SSSP on road grids, whose sources run as single queries side by side:
the grid-wide kernel of such a query takes over from the cluster (forced by a
low hand-over line); bit-exact against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2012_07990_gb300 import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [2, 9, 32])
@pytest.mark.parametrize("hi", ["24", "100000"])
@pytest.mark.parametrize("delta", [400, 6000])
def test_batch(monkeypatch, k, hi, delta):
    from paper_2012_07990_gb300 import g2
    monkeypatch.setenv("G2_CLUSTER_HI", hi)
    g = gg.road_grid(90, seed=3)
    w = gg.pair_weights(g, 1000, seed=1)
    srcs = np.random.default_rng(k).integers(0, g.n, k).astype(np.int32)
    dg = g2.load_graph(g, w)
    dist = torch.full((k, g.n), -7, dtype=torch.int32, device="cuda")
    g2.g2_sssp_batch(dg, srcs, delta, dist)
    got = dist.cpu().numpy()
    for i, s in enumerate(srcs):
        assert np.array_equal(got[i], oracle.sssp(g.n, g.rowptr, g.col, w, int(s))), i
