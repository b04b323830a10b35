"""Adjacency scans by groups of 16 entries and label bytes: lists of every
length from 0 to 70 and around the warp and block limits, whose neighbours'
vertex labels agree in their low byte (1, 257, 513), against the oracle."""
import numpy as np
import pytest

from synth.gfds import GFD, Literal
from synth.graphs import graph_from_edges

from gpu_util import gpu_graph, gpu_run

pytestmark = pytest.mark.gpu

LABELS = [1, 257, 513]


def _graph(reverse):
    """Out-lists (in-lists when reversed) of lengths 0..70, 127..129, 1023..1026, 2100, starting at
    every offset modulo 16, over 2300 neighbours."""
    rng = np.random.default_rng(7 + reverse)
    lengths = list(range(71)) + [127, 128, 129, 1023, 1024, 1025, 1026, 2100] + [1] * 5 + list(range(33, 0, -1))
    n_src, n_dst = len(lengths), 2300
    n = n_src + n_dst
    src, dst = [], []
    for v, d in enumerate(lengths):
        w = n_src + rng.choice(n_dst, size=d, replace=False)
        src += [v] * d
        dst += sorted(int(x) for x in w)
    src, dst = np.array(src), np.array(dst)
    if reverse:
        src, dst = dst, src
    vl = np.array(LABELS)[rng.integers(0, 3, size=n)]
    return graph_from_edges(n, src, dst, rng.integers(0, 3, size=len(src)), vl, rng.integers(0, 4, size=(1, n)))


@pytest.mark.parametrize("reverse", [False, True])
@pytest.mark.parametrize("flags", [0, 0x10])
def test_lists_of_every_length(oracle_mod, reverse, flags):
    g = _graph(reverse)
    dg = gpu_graph(g)
    mode = {"induced": False} if flags else {}
    for a, b in [(1, 257), (257, 1), (513, 513), (-1, 257), (1, -1)]:
        for lab in (-1, 2):
            for edges in ([(0, 1, lab)], [(0, 1, lab), (0, 2, -1)]):
                q = GFD([a, b, 513][: len(edges) + 1], edges, [], [Literal.var(0, 0, 1, 0)])
                if len(edges) == 2 and not reverse and b == -1:
                    continue  # the 2100-list alone has millions of matches
                want = oracle_mod.validate(g, q, **mode)
                nm, v = gpu_run(dg, q, flags=flags)
                assert nm == want[0]
                np.testing.assert_array_equal(v, want[1])
