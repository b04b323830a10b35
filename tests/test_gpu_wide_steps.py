"""Steps that make the second-to-last level grow with what the one before did. Here
the first partial matches have few next candidates (so the steps grow) and the rest
many, so that one step has more of them than rows: those without a row are expanded
where they are made, and when they are too many or too long the call runs again with
steps that have their rows. Counts and tuples against the closed form."""
import numpy as np
import pytest

from synth.gfds import GFD, Literal
from synth.graphs import graph_from_edges

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_2608_02321_gb300")

FEW = 10     # next candidates of the first partial matches
CHUNK = 1024


def _case(low, high, fanout, marked):
    """a -> b -> c: `low` a's point to a b of FEW c's, then `high` a's to one of `fanout` c's, whose first
    `marked` have attribute 1. A b without a's has as many c's as there are a's (so a is matched first)."""
    a, pad = low + high, low + high
    few, many, lone = a, a + 1, a + 2
    c0 = a + 3
    src = np.concatenate([np.arange(a), np.full(FEW, few), np.full(fanout, many), np.full(pad, lone)])
    dst = np.concatenate([np.full(low, few), np.full(high, many), c0 + np.arange(FEW + fanout + pad)])
    n = c0 + FEW + fanout + pad
    label = np.full(n, 2)
    label[:a], label[a:c0] = 0, 1
    attr = np.zeros((1, n))
    attr[0, c0 + FEW:c0 + FEW + marked] = 1
    q = GFD([0, 1, 2], [(0, 1, -1), (1, 2, -1)], [Literal.const(2, 0, 1)], [], True)
    viol = np.stack([np.repeat(np.arange(low, a), marked), np.full(high * marked, many),
                     np.tile(c0 + FEW + np.arange(marked), high)], axis=1)
    return graph_from_edges(n, src, dst, np.zeros(len(src)), label, attr), q, low * FEW + high * fanout, viol


def _session(dg, q):
    s = G.Session(dg, max_slots=2, chunk_rows=CHUNK)
    s.submit(q)
    for _ in range(100000):
        s.step()
        for _, r in s.results():
            return r


# (low, high, fan-out, runs made again): no row for about 5000 of a step's 8192; the
# same with lists over 2^18; 64,000 of 200,000 each, over 2^33 together
CASES = [(3024, 20000, 100, 0), (3024, 5000, 300_000, 1), (10216, 70000, 200_000, 1)]


@pytest.mark.parametrize("low,high,fanout,again", CASES)
@pytest.mark.parametrize("driver", ["persistent", "host_loop", "session"])
def test_more_partial_matches_than_rows(low, high, fanout, again, driver):
    g, q, want, viol = _case(low, high, fanout, 3)
    dg = G.Graph(g)
    if driver == "session":
        r = _session(dg, q)
    else:
        r = dg.validate(q, chunk_rows=CHUNK, flags=G.FLAG_HOST_LOOP if driver == "host_loop" else 0)
    assert r.n_matches == want
    np.testing.assert_array_equal(r.violations(), viol)
    assert r.stat(G.STAT_RERUN) == again


def test_partial_matches_without_a_row_are_counted():
    g, q, want, _ = _case(*CASES[0][:3], 3)
    r = G.Graph(g).validate(q, chunk_rows=CHUNK, flags=G.FLAG_COUNT)
    assert r.n_matches == want and r.counters()["no_row"] > 4000
