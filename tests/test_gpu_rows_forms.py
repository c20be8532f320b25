"""The forms of the tuned multi-source SSSP, each told by its counters and
bit-exact against the oracle: list rounds with hubs longer than a tile, both
forms on directed graphs with weights that differ between an edge's two arcs,
and batches that end just before and just after the last row round, which go on
with the near/far queue from the distances found so far."""
import numpy as np
import pytest

import oracle
from paper_2012_07990_gb300 import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ROUNDS = 32


@pytest.fixture(scope="module")
def g2():
    from paper_2012_07990_gb300 import g2 as m
    return m


def run(g2, g, w, srcs, delta):
    """Distances checked against the oracle; the call's counters."""
    dg = g2.load_graph(g, w)
    dist = torch.full((len(srcs), g.n), -7, dtype=torch.int32, device="cuda")
    g2.g2_set_count_arcs(True)
    try:
        g2.g2_sssp_batch(dg, srcs, delta, dist)
        stats = g2.g2_last_stats()
    finally:
        g2.g2_set_count_arcs(False)
    got = dist.cpu().numpy()
    for i, s in enumerate(srcs):
        assert np.array_equal(got[i], oracle.sssp(g.n, g.rowptr, g.col, w, int(s))), i
    return stats


def arc_weights(g, seed):
    return np.random.default_rng(seed).integers(1, 256, g.m).astype(np.int32)


@pytest.mark.parametrize("k", [1, 8, 9, 16, 17, 32])
@pytest.mark.parametrize("symmetric", [True, False])
def test_list_rounds(g2, k, symmetric):
    """Hubs of 127 .. 2,000 arcs in a chain, leaves shared between neighbours,
    among so many isolated vertices that every frontier is a list."""
    u, v, n, prev = [], [], 0, None
    for leaves in (127, 128, 129, 255, 1023, 1024, 2000):
        at = np.arange(n + 1, n + 1 + leaves)
        u += [np.full(leaves, n)]
        v += [at]
        if prev is not None:
            u += [np.array([prev]), at[::3]]
            v += [np.array([n]), np.full(at[::3].size, prev)]
        prev, n = n, n + 1 + leaves
    g = gg.from_arcs(n + 300000, np.concatenate(u), np.concatenate(v), symmetric=symmetric)
    srcs = np.random.default_rng(k).integers(0, n, k).astype(np.int32)
    srcs[0] = 0
    for delta in (0, 64):
        stats = run(g2, g, arc_weights(g, 5), srcs, delta)
        it = stats["iterations"]
        assert 7 <= it <= ROUNDS
        # a sweep is two launches a round; lists take more
        assert stats["launches"] >= 3 * it


@pytest.mark.parametrize("k", [1, 9, 32])
def test_sweeps_of_a_directed_graph(g2, k):
    rng = np.random.default_rng(2)
    g = gg.from_arcs(500, rng.integers(0, 500, 9000) ** 2 // 500, rng.integers(0, 500, 9000), symmetric=False)
    srcs = rng.integers(0, g.n, k).astype(np.int32)
    for delta in (0, 64):
        stats = run(g2, g, arc_weights(g, 3), srcs, delta)
        assert stats["iterations"] <= ROUNDS


def core_and_tail(tail, symmetric):
    """gnp(400, 0.2) and a path of `tail` vertices behind its vertex 0."""
    core = gg.gnp(400, 0.2, 7)
    u = np.concatenate([np.repeat(np.arange(400), core.degrees()), [0], np.arange(400, 399 + tail)])
    v = np.concatenate([core.col, [400], np.arange(401, 400 + tail)])
    return gg.from_arcs(400 + tail, u, v, symmetric=symmetric)


@pytest.mark.parametrize("symmetric", [True, False])
@pytest.mark.parametrize("k", [1, 9, 32])
@pytest.mark.parametrize("tail", [30, 31, 32, 33, 60, 300])
def test_batches_about_the_last_row_round(g2, symmetric, k, tail):
    """All sources at the head of the tail.  With unit weights a vertex's distance
    falls once: a round a hop, and every arc is relaxed in one round."""
    g = core_and_tail(tail, symmetric)
    srcs = np.zeros(k, np.int32)
    unit = np.ones(g.m, np.int32)
    for w in (unit, arc_weights(g, 4)):
        for delta in (0, 64):
            stats = run(g2, g, w, srcs, delta)
            if w is unit:
                assert stats["iterations"] == tail + 1
                # no vertex's arcs are relaxed once more by what follows the rows
                assert stats["arcs_examined"] == g.m


@pytest.mark.parametrize("tail", [3, 60])
@pytest.mark.parametrize("last, over", [(2**31 - 4, False), (2**31 - 3, True)])
@pytest.mark.parametrize("delta", [0, 64])
def test_overflow_is_told_in_either_form(g2, tail, last, over, delta):
    """A hub with 40 leaves, unit arcs but 0 -> 40 of weight `last`: from leaf 1
    vertex 40 lies at last + 1, and its arc back leads to last + 2, which may
    not reach INT32_MAX; behind the hub a tail."""
    u = np.concatenate([np.zeros(40, int), [0], np.arange(41, 40 + tail)])
    v = np.concatenate([np.arange(1, 41), [41], np.arange(42, 41 + tail)])
    g = gg.from_arcs(41 + tail, u, v)
    src = np.repeat(np.arange(g.n), g.degrees())
    w = np.ones(g.m, np.int32)
    w[(src == 0) & (g.col == 40)] = last
    dg = g2.load_graph(g, w)
    dist = torch.empty((1, g.n), dtype=torch.int32, device="cuda")
    if over:
        with pytest.raises(g2.G2Error) as e:
            g2.g2_sssp_batch(dg, [1], delta, dist)
        assert e.value.status == g2.G2_EOVERFLOW
    else:
        g2.g2_sssp_batch(dg, [1], delta, dist)
        want = np.full(g.n, 2)
        want[[0, 1, 40]] = [1, 0, last + 1]
        want[41:] = 2 + np.arange(tail)
        assert np.array_equal(dist.cpu().numpy()[0], want)


@pytest.mark.parametrize("k", [1, 5, 32])
@pytest.mark.parametrize("delta", [0, 300])
def test_frontier_that_does_not_fall(g2, k, delta):
    """A band 50 hops across: given up at the look, with most vertices flagged."""
    rng = np.random.default_rng(6)
    i = np.repeat(np.arange(4000), 20)
    j = i + rng.integers(1, 80, i.size)
    g = gg.from_arcs(4000, i[j < 4000], j[j < 4000])
    srcs = rng.integers(0, g.n, k).astype(np.int32)
    srcs[0] = 0
    run(g2, g, gg.pair_weights(g, 255, seed=2), srcs, delta)
