"""Large launches of the adjacency scans take larger work units than small ones
and share equal refinements between GFDs: a batch large enough for the large
units gives the candidates, index sizes, matches and violations that its GFDs
give one call at a time."""
import numpy as np
import pytest

from synth import configs

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_2608_02321_gb300")


@pytest.mark.parametrize("flags", [0, 0x10, 0x20])
def test_batch_units_equal_single(flags):
    g, qs = configs.batched(scale=10, n_gfds=128)
    # patterns whose edges nearly all carry labels keep the match counts small
    for i, q in enumerate(qs):
        q.edges = [(a, b, l if l >= 0 else (i + a) % 32) for a, b, l in q.edges]
    dg = G.Graph(g)
    opts = dict(flags=flags, frontier_budget_bytes=8 << 30)
    batch = dg.validate_batch(qs, max_violations_hint=1 << 22, **opts)
    lists = G.violations_all(batch)
    for q, b, v in zip(qs, batch, lists):
        r = dg.validate(q, **opts)
        assert b.n_matches == r.n_matches, q.name
        assert b.stat(G.STAT_CANDIDATES) == r.stat(G.STAT_CANDIDATES), q.name
        assert b.stat(G.STAT_INDEX) == r.stat(G.STAT_INDEX), q.name
        np.testing.assert_array_equal(v, r.violations(), err_msg=q.name)
