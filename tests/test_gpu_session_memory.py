"""A session's budget counts what its running requests hold: their index edges as
they are, not the bound known before they are counted, so requests keep joining."""
import numpy as np
import pytest

from synth.gfds import GFD
from synth.graphs import graph_from_edges

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_2608_02321_gb300")


def test_requests_join_while_index_edges_are_few():
    n, m = 200_000, 4_000_000
    rng = np.random.default_rng(5)
    key = np.unique(rng.integers(0, n, m) * n + rng.integers(0, n, m))
    src, dst = key // n, key % n
    src, dst = src[src != dst], dst[src != dst]
    label = np.full(n, 1)
    label[0] = 0   # one root: a few thousand index edges, bounded by 12 bytes for each of the graph's edges
    dg = G.Graph(graph_from_edges(n, src, dst, np.zeros(len(src)), label, np.zeros((1, n))))
    q = GFD([0, -1, -1, -1, 1], [(0, 1, -1), (1, 2, -1), (2, 3, -1)])   # and a node apart: many steps
    want = dg.validate(q).n_matches
    assert want > 10 ** 8
    # two requests fit at their bounds (52 MB each), five at what they hold
    s = G.Session(dg, max_slots=8, frontier_budget_bytes=120_000_000, chunk_rows=1024, max_violations_hint=1024)
    ids = [s.submit(q) for _ in range(5)]
    most, got = 0, {}
    for _ in range(100000):
        _, running, queued = s.step()
        most = max(most, running)
        got.update((i, r.n_matches) for i, r in s.results())
        if not running and not queued:
            break
    assert got == {i: want for i in ids}
    assert most >= 4
