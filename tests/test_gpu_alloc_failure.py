"""Calls on a device without room: each allocation of a call fails in turn.
The call reports G2_ENOMEM or goes on without that buffer, and the next call on
the same handle is right."""
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


def fail_each(g2, dg, call, min_bytes=0):
    """call(handle) with the first, second, ... of its allocations failing, on a
    handle of its own each time; yields the handle and whether the call got by."""
    for nth in range(1, 100):
        view = dg.view()
        g2.g2_diag_fail_alloc(nth, min_bytes)
        status = g2.G2_OK
        try:
            call(view)
        except g2.G2Error as e:
            status = e.status
        if g2.g2_diag_fail_alloc(0):        # it makes fewer allocations
            assert status == g2.G2_OK and nth > 1
            return
        assert status in (g2.G2_OK, g2.G2_ENOMEM)
        yield view, status == g2.G2_OK
    pytest.fail("a call with 100 allocations")


def test_next_call_is_right(g2):
    g = gg.rmat(10, seed=2)
    want = oracle.bfs(g.n, g.rowptr, g.col, 3, False)[0]
    dg = g2.load_graph(g)
    depth = torch.empty(g.n, dtype=torch.int32, device="cuda")

    def bfs(h):
        g2.g2_bfs(h, 3, depth, None, g2.schedule("STRICT"))

    for view, ok in fail_each(g2, dg, bfs):
        if not ok:
            depth.fill_(-9)
            bfs(view)
        assert np.array_equal(depth.cpu().numpy(), want)


@pytest.mark.parametrize("k", [1, 9, 32])
def test_sssp_batch_goes_on_without_rows(g2, k):
    """The tuned multi-source SSSP survives each single failed allocation: it
    goes on without the distance rows."""
    g = gg.rmat(10, seed=3)
    w = gg.pair_weights(g, 255, seed=1)
    srcs = np.random.default_rng(k).integers(0, g.n, k).astype(np.int32)
    want = np.stack([oracle.sssp(g.n, g.rowptr, g.col, w, int(s)) for s in srcs])
    dist = torch.empty((k, g.n), dtype=torch.int32, device="cuda")
    failed = []
    for nth in range(1, 40):
        dg = g2.load_graph(g, w)
        dist.fill_(-9)
        g2.g2_diag_fail_alloc(nth)
        g2.g2_sssp_batch(dg, srcs, 64, dist)
        left = g2.g2_diag_fail_alloc(0)
        assert np.array_equal(dist.cpu().numpy(), want), nth
        if left:
            break
        failed.append(nth)
        g2.g2_sssp_batch(dg, srcs, 64, dist)
        assert np.array_equal(dist.cpu().numpy(), want), nth
    assert len(failed) >= 8       # counters, rows, sources of the arcs, flags, list, degrees, scan


@pytest.mark.parametrize("k", [17, 33, 64])
def test_bfs_batch_goes_on_without_planes(g2, k):
    g = gg.rmat(10, seed=3)
    srcs = np.random.default_rng(k).integers(0, g.n, k).astype(np.int32)
    want = np.stack([oracle.bfs(g.n, g.rowptr, g.col, int(s), False)[0] for s in srcs])
    dg = g2.load_graph(g)
    depth = torch.empty((k, g.n), dtype=torch.int32, device="cuda")
    depth.fill_(-9)
    g2.g2_diag_fail_alloc(1, 40 * g.n)       # the planes: no other buffer is as large
    g2.g2_bfs_batch(dg, srcs, depth)
    assert g2.g2_diag_fail_alloc(0) == 0
    assert np.array_equal(depth.cpu().numpy(), want)


def test_edge_blocking_is_all_or_nothing(g2):
    """A rebuild that fails leaves no layout of another segment size behind: the
    next request of the size before it builds, and its export is what it was."""
    g = gg.rmat(9, seed=1)
    dg = g2.load_graph(g)

    def export():
        ns = g2.g2_edge_block(dg, 100)
        s, d = (torch.full((g.m,), -1, dtype=torch.int32, device="cuda") for _ in range(2))
        seg = torch.full((ns + 1,), -1, dtype=torch.int64, device="cuda")
        g2.g2_edge_block_export(dg, s, d, seg)
        return [x.cpu().numpy() for x in (s, d, seg)]

    want = export()
    for nth in range(1, 20):
        g2.g2_diag_fail_alloc(nth)
        try:
            g2.g2_edge_block(dg, 60)
        except g2.G2Error as e:
            assert e.status == g2.G2_ENOMEM
        if g2.g2_diag_fail_alloc(0):
            break
        for a, b in zip(export(), want):
            assert np.array_equal(a, b), nth
    assert nth >= 7          # six arrays and the scan's


@pytest.mark.parametrize("kernel", ["seg", "blk", "merge"])
def test_pagerank_layouts_are_all_or_nothing(g2, monkeypatch, kernel):
    """PageRank on a graph whose layout could not be built builds it on the next
    call."""
    monkeypatch.setenv("G2_PR_KERNEL", kernel)
    g = gg.rmat(9, seed=1)
    want = oracle.pagerank_graph(g, 0.85, 5)
    rank = torch.empty(g.n, dtype=torch.float32, device="cuda")
    for nth in range(1, 60):
        dg = g2.load_graph(g)
        g2.g2_diag_fail_alloc(nth)
        try:
            g2.g2_pagerank(dg, 0.85, 5, rank)
        except g2.G2Error as e:
            assert e.status == g2.G2_ENOMEM
        if g2.g2_diag_fail_alloc(0):
            break
        rank.fill_(-1)
        g2.g2_pagerank(dg, 0.85, 5, rank)
        assert np.abs(rank.cpu().numpy().astype(np.float64) - want).sum() <= 1e-5, nth
    assert nth > 4
