"""Batches whose refinement results and marks are too many to lie apart: results take
the places of bitmaps that are no longer read, and come out as each GFD's alone; and
their memory stays near that of the levels' final bitmaps and ranks."""
import gc

import numpy as np
import pytest

from synth.gfds import GFD
from synth.graphs import graph_from_edges

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_2608_02321_gb300")
torch = pytest.importorskip("torch")


def _graph(n, m, label, seed):
    rng = np.random.default_rng(seed)
    key = np.unique(rng.integers(0, n, m) * n + (n * rng.random(m) ** 2).astype(np.int64))
    src, dst = key // n, key % n
    keep = src != dst
    return graph_from_edges(n, src[keep], dst[keep], np.zeros(int(keep.sum())), label, np.zeros((1, n)))


def _pattern(rng, k, label, cycle):
    skel = [(u - 1 if cycle else int(rng.integers(0, u)), u) for u in range(1, k)] + ([(k - 1, 0)] if cycle else [])
    return GFD([label() for _ in range(k)], [(a, b, -1) if rng.random() < 0.5 else (b, a, -1) for a, b in skel])


@pytest.mark.parametrize("flags", [0, G.FLAG_NON_INDUCED])
def test_results_as_alone(flags):
    n = 1_000_000
    rng = np.random.default_rng(3)
    p = 1.0 / np.arange(1, 13)
    dg = G.Graph(_graph(n, 3_000_000, rng.choice(12, size=n, p=p / p.sum()), 4))
    qs = [_pattern(rng, int(rng.integers(4, 9)), lambda: int(rng.integers(-1, 12)), i % 4 == 3) for i in range(400)]
    batch = dg.validate_batch(qs, chunk_rows=4096, flags=flags)   # 400 x 6 levels x 125 KB at least
    for i, (q, b) in enumerate(zip(qs, batch)):
        one = dg.validate(q, chunk_rows=4096, flags=flags)
        for what in (G.STAT_CANDIDATES, G.STAT_INDEX):
            assert b.stat(what) == one.stat(what), i
        assert b.n_matches == one.n_matches, i
    assert sum(b.n_matches for b in batch) > 0


def test_memory_of_many_refinements():
    gc.collect()
    n, k = 4_000_000, 8
    rng = np.random.default_rng(6)
    p = np.tile([1.0, 8.0], 500)
    dg = G.Graph(_graph(n, 4_000_000, rng.choice(1000, size=n, p=p / p.sum()), 7))
    qs = [_pattern(rng, k, lambda: int(rng.integers(0, 1000)), i % 2 == 1) for i in range(128)]
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    dg.validate_batch(qs, chunk_rows=1024, max_violations_hint=1024)
    torch.cuda.synchronize()
    used = before - torch.cuda.mem_get_info()[0]
    keys = {(q.node_label[u], sum(a == u for a, _, _ in q.edges), sum(b == u for _, b, _ in q.edges))
            for q in qs for u in range(k)}
    levels, bitmap = len(qs) * k, n // 8
    # a filter bitmap per key; a final bitmap and a rank per level; half a level's more
    # for what a phase reads and writes; lists, index and rows below 128 MB
    assert used <= (2.5 * levels + len(keys)) * bitmap + (128 << 20)
