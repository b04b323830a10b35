"""A call on a device that is nearly full: room for index edges at their bound is
given up before the call is refused."""
import gc

import numpy as np
import pytest

from synth.gfds import GFD
from synth.graphs import graph_from_edges

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_2608_02321_gb300")
torch = pytest.importorskip("torch")


def test_index_edges_are_counted_when_their_bound_does_not_fit():
    n, m = 200_000, 10_000_000
    rng = np.random.default_rng(8)
    key = np.unique(rng.integers(0, n, m) * n + rng.integers(0, n, m))
    src, dst = key // n, key % n
    keep = src != dst
    label = np.full(n, 1)
    label[0] = 0
    # one root; each of three index edges bounded by the graph's edges (80, 80 and 40 MB)
    q = GFD([0, -1, -1, -1, -1], [(0, 1, -1), (1, 2, -1), (2, 3, -1), (3, 4, -1)])
    opts = {"frontier_budget_bytes": 4 << 20, "max_violations_hint": 1 << 10}
    g = graph_from_edges(n, src[keep], dst[keep], np.zeros(int(keep.sum())), label, np.zeros((1, n)))
    want = G.Graph(g).validate(q, **opts).n_matches
    assert want > 1_000_000
    gc.collect()
    torch.cuda.empty_cache()
    dg = G.Graph(g)
    dg.validate(GFD([0], []), **opts)   # the kernels and the pool are there
    torch.cuda.synchronize()
    filler = torch.empty(torch.cuda.mem_get_info()[0] - (160 << 20), dtype=torch.uint8, device="cuda")
    try:
        assert dg.validate(q, **opts).n_matches == want
    finally:
        del filler
        torch.cuda.empty_cache()
    assert dg.validate(q, **opts).n_matches == want
