"""Graphs with many attributes: their columns are reordered a few at a time, and a
graph whose attributes fill most of the free memory still loads."""
import gc

import numpy as np
import pytest

from synth.gfds import GFD, Literal
from synth.graphs import graph_from_edges

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_2608_02321_gb300")
torch = pytest.importorskip("torch")


def _graph(n, n_attrs):
    """A ring; attribute a of vertex v is (v + 7 a) % 1000."""
    v = np.arange(n, dtype=np.int32)
    attrs = np.empty((n_attrs, n), dtype=np.int32)
    for a in range(n_attrs):
        attrs[a] = (v + 7 * a) % 1000
    return graph_from_edges(n, v, (v + 1) % n, np.zeros(n), v % 5, attrs)


def _check(dg, n, a):
    """x -> y with x.a = 0: x = -7 a (mod 1000), and y.a is 1 then."""
    q = GFD([-1, -1], [(0, 1, -1)], [Literal.const(0, a, 0)], [Literal.const(1, a, 2)])
    r = dg.validate(q, frontier_budget_bytes=1 << 20, max_violations_hint=1 << 16)
    x = np.arange(-7 * a % 1000, n, 1000)
    assert r.n_matches == n
    np.testing.assert_array_equal(r.violations(), np.stack([x, (x + 1) % n], axis=1))


@pytest.mark.parametrize("n,n_attrs", [(1000, 1), (500_000, 140), (500_000, 134), (500_000, 135)])
def test_every_column(n, n_attrs):
    g = _graph(n, n_attrs)   # 134 columns of 500,000 at a time
    dg = G.Graph(g)
    for a in {0, n_attrs // 2, n_attrs - 1, min(133, n_attrs - 1), min(134, n_attrs - 1)}:
        _check(dg, n, a)


def test_attributes_that_fill_the_memory():
    gc.collect()
    torch.cuda.empty_cache()
    n, n_attrs = 1_000_000, 600   # 2.4 GB
    g = _graph(n, n_attrs)
    free = torch.cuda.mem_get_info()[0]
    filler = torch.empty(free - (3 << 30) - (512 << 20), dtype=torch.uint8, device="cuda")
    try:
        dg = G.Graph(g)
        del filler
        _check(dg, n, 599)
    finally:
        torch.cuda.empty_cache()
