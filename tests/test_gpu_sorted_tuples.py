"""Sorted violation tuples around the limits of the two sorts (ranking up to 2^26
pairs of tuples, radix sort of packed keys beyond): all ordered selections of a
star's leaves, one result at a time and several together, in id ranges whose
bits split a 64-bit key between columns."""
import itertools

import numpy as np
import pytest

from synth.gfds import GFD
from synth.graphs import graph_from_edges

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_2608_02321_gb300")


def _star(n, leaves, seed):
    rng = np.random.default_rng(seed)
    ids = rng.choice(n, size=leaves + 1, replace=False)
    g = graph_from_edges(n, np.full(leaves, ids[0]), ids[1:], np.zeros(leaves), np.zeros(n), np.zeros((1, n)))
    return G.Graph(g), int(ids[0]), np.sort(ids[1:])


def _query(arms):
    return GFD([-1] * (arms + 1), [(0, 1 + j, -1) for j in range(arms)], [], [], True)


def _want(center, leaves, arms):
    p = np.array(list(itertools.permutations(leaves.tolist(), arms)), dtype=np.int32).reshape(-1, arms)
    return np.concatenate([np.full((len(p), 1), center, dtype=np.int32), p], axis=1)


@pytest.mark.parametrize("n", [200, 70_001, 1 << 22])
@pytest.mark.parametrize("leaves,arms", [(1, 1), (33, 1), (91, 2), (92, 2), (20, 4), (8, 6)])
def test_single_and_together(n, leaves, arms):
    dg, center, ids = _star(n, leaves, 5)
    want = _want(center, ids, arms)
    r = dg.validate(_query(arms))
    assert r.n_matches == len(want)
    np.testing.assert_array_equal(r.violations(), want)
    # together with results of other widths, some empty
    others = [a for a in (1, 2, 3) if leaves ** a < 50_000]
    qs = [_query(a) for a in others] + [GFD([5], [], [], [], True), _query(arms)]
    lists = G.violations_all(dg.validate_batch(qs))
    for a, v in zip(others, lists):
        np.testing.assert_array_equal(v, _want(center, ids, a) if leaves >= a else np.empty((0, a + 1), np.int32))
    assert lists[len(others)].shape == (0, 1)
    np.testing.assert_array_equal(lists[-1], want)
