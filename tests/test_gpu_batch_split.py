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


def test_queries_side_by_side(monkeypatch):
    """SSSP and BC from several threads, each on a view and a stream of its own,
    in the grid-wide kernels; the same results as one after another."""
    import threading
    from paper_2012_07990_gb300 import g2
    monkeypatch.setenv("G2_CLUSTER_HI", "24")
    monkeypatch.setenv("G2_CLUSTER_BC_HI", "24")
    g = gg.road_grid(90, seed=3)
    w = gg.pair_weights(g, 1000, seed=1)
    srcs = np.random.default_rng(4).integers(0, g.n, 24)
    dg = g2.load_graph(g, w)
    wm = g2.schedule("WM", kernel_fusion=True)
    dist = torch.full((24, g.n), -7, dtype=torch.int32, device="cuda")
    bc = torch.zeros((24, g.n), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    errors = []

    def work(t):
        try:
            view = dg.view()
            with torch.cuda.stream(torch.cuda.Stream()):
                for i in range(t, 24, 6):
                    g2.g2_sssp_delta(view, int(srcs[i]), 3000, dist[i], wm)
                    g2.g2_bc(view, [srcs[i]], bc[i], wm)
        except Exception as e:
            errors.append(e)

    threads = [threading.Thread(target=work, args=(t,)) for t in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors
    one = torch.empty(g.n, dtype=torch.float64, device="cuda")
    for i, s in enumerate(srcs):
        assert np.array_equal(dist[i].cpu().numpy(), oracle.sssp(g.n, g.rowptr, g.col, w, int(s))), i
        g2.g2_bc(dg, [s], one, wm)
        want, got = one.cpu().numpy(), bc[i].cpu().numpy()
        assert np.all(np.abs(got - want) <= 1e-6 * np.abs(want) + 1e-12 * np.abs(want).max())
