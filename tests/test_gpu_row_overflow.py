"""Steps of the fused levels take more work items than their row buffers hold:
partial matches that find no row are expanded where they are made. A star of
many leaves whose last level has more than 64 candidates per partial match, with
the smallest row buffers, alone and in batches large enough for the large
buffers, against closed forms."""
import math

import numpy as np
import pytest

from synth.gfds import GFD
from synth.graphs import graph_from_edges

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_2608_02321_gb300")


def _stars(hubs, leaves):
    """`hubs` disjoint out-stars."""
    n = hubs * (leaves + 1)
    src = np.repeat(np.arange(hubs) * (leaves + 1), leaves)
    dst = src + np.tile(np.arange(1, leaves + 1), hubs)
    return graph_from_edges(n, src, dst, np.zeros(len(src)), np.zeros(n), np.zeros((1, n)))


@pytest.mark.parametrize("leaves,arms", [(65, 2), (120, 2), (90, 3), (66, 3)])
@pytest.mark.parametrize("flags", [0, G.FLAG_HOST_LOOP])
def test_no_row_left(leaves, arms, flags):
    hubs = 40
    dg = G.Graph(_stars(hubs, leaves))
    q = GFD([-1] * (arms + 1), [(0, 1 + j, -1) for j in range(arms)])
    want = hubs * math.perm(leaves, arms)
    for chunk in (1024, 4096, 0):
        assert dg.validate(q, chunk_rows=chunk, flags=flags).n_matches == want


def test_large_buffers_of_a_batch():
    hubs, leaves = 30, 150
    dg = G.Graph(_stars(hubs, leaves))
    qs = [GFD([-1] * (a + 1), [(0, 1 + j, -1) for j in range(a)]) for a in [1, 2] * 6 + [3, 3]]
    # 2^16 rows per level and GFD are the least that large buffers are used for
    for budget in (0, 200 << 20, 24 << 20):
        res = dg.validate_batch(qs, frontier_budget_bytes=budget)
        for q, r in zip(qs, res):
            assert r.n_matches == hubs * math.perm(leaves, q.k - 1)
