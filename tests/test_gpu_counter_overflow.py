"""A step whose new partial matches have more than 2^40 next candidates together
cannot be counted: the call ends with GFD_ERR_OVERFLOW in its first step, and the
graph stays usable."""
import numpy as np
import pytest

from synth.gfds import GFD
from synth.graphs import graph_from_edges

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_2608_02321_gb300")


@pytest.mark.parametrize("flags", [0, G.FLAG_HOST_LOOP])
def test_fan_outs_beyond_the_counter(flags):
    n, m = 1_200_000, 1_050_000   # a path of m edges: m rows x -> y with n candidates z each, 1.26e12 > 2^40
    src = np.arange(m)
    dg = G.Graph(graph_from_edges(n, src, src + 1, np.zeros(m), np.zeros(n), np.zeros((1, n))))
    with pytest.raises(G.GfdError) as e:
        dg.validate(GFD([-1, -1, -1], [(0, 1, -1)]), flags=flags)
    assert e.value.code == G.GFD_ERR_OVERFLOW
    assert "chunk_rows" in str(e.value)
    assert dg.validate(GFD([-1, -1], [(0, 1, -1)]), flags=flags).n_matches == m
