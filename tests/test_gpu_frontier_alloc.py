"""Frontiers after a call that failed: a sparse one whose list could not grow is
empty, has no list, and works again as a target, an output and an input; the
output of a round that failed is what it was, also where it is the input."""
import numpy as np
import pytest

from paper_2012_07990_gb300 import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g2():
    from paper_2012_07990_gb300 import g2 as m
    return m


def members(f, room):
    out = torch.empty(room, dtype=torch.int32, device="cuda")
    k = f.to_list(out)
    return np.sort(out[:k].cpu().numpy())


@pytest.mark.parametrize("then", ["VERTEX_BASED", "STRICT", "ETWC", "as output"])
def test_frontier_whose_list_could_not_grow(g2, then):
    g = gg.star(50)
    dg = g2.load_graph(g)
    f, other, hub = (g2.g2_frontier_create(dg, g2.G2_FRONTIER_SPARSE) for _ in range(3))
    many = np.zeros(200, np.int32)
    other.set(many)                                  # the workspace has room for 200 from here on
    hub.set([0])
    f.set([3, 4])
    g2.g2_diag_fail_alloc(1, 4 * many.size)
    with pytest.raises(g2.G2Error) as e:
        f.set(many)
    assert g2.g2_diag_fail_alloc(0) == 0 and e.value.status == g2.G2_ENOMEM
    assert f.size() == 0 and members(f, 50).size == 0
    val = torch.arange(50, dtype=torch.int32, device="cuda")
    if then == "as output":
        assert g2.g2_edgeset_apply(dg, g2.G2_OP_LABEL_MIN, hub, val, None, None, f) == 49
        assert np.array_equal(members(f, 50), np.arange(1, 50))
    else:
        assert g2.g2_edgeset_apply(dg, g2.G2_OP_LABEL_MIN, f, val, None, g2.schedule(then), other) == 0
        assert np.array_equal(val.cpu().numpy(), np.arange(50))
    f.set(many)
    assert f.size() == 200


@pytest.mark.parametrize("fmt", ["G2_FRONTIER_SPARSE", "G2_FRONTIER_BITMAP"])
@pytest.mark.parametrize("lb", ["VERTEX_BASED", "STRICT", "ETWC"])
@pytest.mark.parametrize("same", [False, True])
def test_output_of_a_failed_round(g2, fmt, lb, same):
    g = gg.star(300)
    dg = g2.load_graph(g, np.full(g.m, 100, np.int32))
    fin, other = (g2.g2_frontier_create(dg, getattr(g2, fmt)) for _ in range(2))
    fout = fin if same else other
    fin.set([0, 7])
    if not same:
        fout.set([3, 4, 5])
    before = members(fout, 300)
    dist = torch.full((300,), 2**31 - 50, dtype=torch.int32, device="cuda")   # 100 more is too far
    with pytest.raises(g2.G2Error) as e:
        g2.g2_edgeset_apply(dg, g2.G2_OP_RELAX_MIN, fin, dist, None, g2.schedule(lb), fout)
    assert e.value.status == g2.G2_EOVERFLOW
    assert fout.size() == before.size and np.array_equal(members(fout, 300), before)
    assert np.array_equal(members(fin, 300), [0, 7])
    # and a round that does not fail, twice: the lists change hands
    for _ in range(2):
        fin.set([0])
        val = torch.arange(300, dtype=torch.int32, device="cuda")
        assert g2.g2_edgeset_apply(dg, g2.G2_OP_LABEL_MIN, fin, val, None, g2.schedule(lb), fout) == 299
        assert np.array_equal(members(fout, 300), np.arange(1, 300))
        if not same:
            assert np.array_equal(members(fin, 300), [0])
