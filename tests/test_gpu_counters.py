"""The counting pass against counts known from the graph: absent edges are counted up
to the first that is there, and the last level's look into a row filter is a load
and, when it refuses the candidate, a settled check. Checks are settled or searched;
the statistic of pairs tested is the same with and without counting."""
import numpy as np
import pytest

from synth.gfds import GFD
from synth.graphs import graph_from_edges

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_2608_02321_gb300")


def _counters(dg, q, flags=0, matches=0):
    r = dg.validate(q, flags=flags | G.FLAG_COUNT)
    assert r.n_matches == matches
    c = r.counters()
    assert c["checks"] == c["sig_settled"] + c["searches"]
    assert dg.validate(q, flags=flags).stat(G.STAT_PROBES) == r.stat(G.STAT_PROBES) >= c["checks"]
    return c


@pytest.mark.parametrize("leaves", [40, 100])   # the last level within the step before, and from stored rows
def test_absent_edges_up_to_the_first_found(leaves):
    """An out-star whose leaves a < b are joined a -> b, and two arms that must not be: of the ordered pairs
    (first arm, second arm), half have the edge second -> first, looked at second, half the other, looked at third."""
    a, b = np.triu_indices(leaves, 1)
    src, dst = np.concatenate([np.zeros(leaves), a + 1]), np.concatenate([np.arange(leaves), b]) + 1
    label = np.ones(leaves + 1)
    label[0] = 0
    dg = G.Graph(graph_from_edges(leaves + 1, src, dst, np.zeros(len(src)), label, np.zeros((1, leaves + 1))))
    c = _counters(dg, GFD([0, 1, 1], [(0, 1, -1), (0, 2, -1)]))
    pairs = leaves * (leaves - 1)
    assert c["items"] == leaves + leaves * leaves and c["items_last"] == leaves * leaves
    assert c["neg_checks"] == leaves + pairs // 2 * 2 + pairs // 2 * 3
    assert c["neg_checks"] <= c["checks"] <= leaves + pairs * 3


def test_the_first_look_at_the_last_level():
    """Two hubs -> 20 leaves -> 30 ends each, and a triangle hub, leaf, leaf that is nowhere: every pair of
    leaves is looked up in the first leaf's row filter, which lets few pass (one bit in eight is set)."""
    leaves, ends = 20, 30
    n = 2 + leaves + leaves * ends
    leaf = 2 + np.arange(leaves)
    src = np.concatenate([np.zeros(leaves), np.ones(leaves), np.repeat(leaf, ends)])
    dst = np.concatenate([leaf, leaf, np.arange(2 + leaves, n)])
    label = np.full(n, 2)
    label[:2], label[2:2 + leaves] = 0, 1
    dg = G.Graph(graph_from_edges(n, src, dst, np.zeros(len(src)), label, np.zeros((1, n))))
    c = _counters(dg, GFD([0, 1, 1], [(0, 1, -1), (0, 2, -1), (1, 2, -1)]), G.FLAG_NO_REFINE)
    assert c["items_last"] == 2 * leaves * leaves
    assert c["sig_loads"] >= c["items_last"]
    assert c["checks"] >= c["items_last"] // 2 and c["sig_settled"] >= c["items_last"] // 2
