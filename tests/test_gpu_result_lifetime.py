"""Results dropped unread while the kernel that writes their violation lists may
still be queued: their memory goes back to the graph's pool only after it, so calls
on other streams (and the end of the graph) that take the memory over stay exact."""
import math

import numpy as np
import pytest

from synth.gfds import GFD
from synth.graphs import graph_from_edges

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_2608_02321_gb300")
torch = pytest.importorskip("torch")

LEAVES = 1500


def _graph():
    src, dst = np.zeros(LEAVES), np.arange(1, LEAVES + 1)
    return graph_from_edges(LEAVES + 1, src, dst, np.zeros(LEAVES), np.zeros(LEAVES + 1), np.zeros((1, LEAVES + 1)))


@pytest.mark.parametrize("batch", [1, 3])
def test_unread_results_and_another_stream(batch):
    star = GFD([-1] * 3, [(0, 1, -1), (0, 2, -1)], [], [], True)   # 2.2M violations
    edge = GFD([-1] * 2, [(0, 1, -1)], [], [], True)
    pairs = np.stack([np.zeros(LEAVES), np.arange(1, LEAVES + 1)], axis=1)
    other = torch.cuda.Stream()
    opts = {"max_violations_hint": 3 * batch * LEAVES * LEAVES, "frontier_budget_bytes": 32 << 20}
    for _ in range(4):
        dg = G.Graph(_graph())
        for _ in range(5):
            counts = [r.n_violations for r in dg.validate_batch([star] * batch, **opts)]   # dropped here
            got = dg.validate(edge, stream=other, frontier_budget_bytes=32 << 20, max_violations_hint=1 << 20)
            assert counts == [math.perm(LEAVES, 2)] * batch
            np.testing.assert_array_equal(got.violations(), pairs)
        last = dg.validate_batch([star] * batch, **opts)
        del dg, got, last   # the graph goes while its last call's lists may still be written


def test_unread_results_do_not_pile_up():
    """What was dropped unread is free for the next call."""
    star = GFD([-1] * 3, [(0, 1, -1), (0, 2, -1)], [], [], True)   # a list of 27 MB
    dg = G.Graph(_graph())
    opts = {"max_violations_hint": LEAVES * LEAVES, "frontier_budget_bytes": 32 << 20}
    for _ in range(3):
        dg.validate(star, **opts)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    for _ in range(30):
        assert dg.validate(star, **opts).n_violations == math.perm(LEAVES, 2)
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] <= 64 << 20
