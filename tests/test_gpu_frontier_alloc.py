"""A sparse frontier whose list could not grow: it is empty, has no list, and
works again as a target, an output and an input."""
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
