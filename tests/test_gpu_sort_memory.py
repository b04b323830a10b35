"""The device memory that sorting a long violation list needs is given back: the
graph's pool keeps at most 64 MiB more than it held before."""
import gc
import math

import numpy as np
import pytest

from synth.gfds import GFD
from synth.graphs import graph_from_edges

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_2608_02321_gb300")
torch = pytest.importorskip("torch")

LEAVES = 4000


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("together", [False, True])
def test_scratch_is_given_back(together):
    gc.collect()
    src, dst = np.zeros(LEAVES), np.arange(1, LEAVES + 1)
    dg = G.Graph(graph_from_edges(LEAVES + 1, src, dst, np.zeros(LEAVES), np.zeros(LEAVES + 1), np.zeros((1, LEAVES + 1))))
    n = math.perm(LEAVES, 2)
    r = dg.validate(GFD([-1] * 3, [(0, 1, -1), (0, 2, -1)], [], [], True), frontier_budget_bytes=16 << 20,
                    max_violations_hint=n)
    before = _free()
    for _ in range(2):
        v = G.violations_all([r])[0] if together else r.violations()
        assert v.shape == (n, 3) and (v[0] == (0, 1, 2)).all() and (v[-1] == (0, LEAVES, LEAVES - 1)).all()
        assert before - _free() <= 80 << 20   # 64 MiB and the pool's rounding; the sort takes 0.5 GB
