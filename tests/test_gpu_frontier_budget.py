"""A call's partial-match buffers, large ones included, stay inside the frontier
budget that it was given."""
import gc

import numpy as np
import pytest

from synth.gfds import GFD
from synth.graphs import graph_from_edges

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_2608_02321_gb300")
torch = pytest.importorskip("torch")

BUDGET = 8 << 30
SLACK = 64 << 20  # slot tables, bitmaps and index of a tiny graph, rounding of the pool


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("n", [1, 8, 9, 10, 11, 12, 13, 16, 40])
def test_budget_is_kept(n):
    gc.collect()
    src = np.arange(30)
    dg = G.Graph(graph_from_edges(31, src, src + 1, np.zeros(30), np.zeros(31), np.zeros((1, 31))))
    q = GFD([-1] * 4, [(0, 1, -1), (1, 2, -1), (2, 3, -1)])
    before = _free()
    res = dg.validate_batch([q] * n, frontier_budget_bytes=BUDGET, max_violations_hint=1024)
    assert [r.n_matches for r in res] == [28] * n
    used = before - _free()
    assert used <= BUDGET + SLACK
    # three quarters at least (rows are at most 15.7M per level and GFD)
    assert used >= min(BUDGET * 3 // 4, n * 15_000_000 * 80)
