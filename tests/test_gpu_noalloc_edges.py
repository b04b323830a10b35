"""gfd_node_candidates_noalloc at the edges of its tiles: vertex counts around
a lane's four vertices, a warp's 128, a block's round of 1024 and the switch
from one round per tile to eight (tiles of 8192)."""
import numpy as np
import pytest

from synth.gfds import GFD
from synth.graphs import Graph

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_2608_02321_gb300")
torch = pytest.importorskip("torch")

SIZES = [1, 3, 4, 5, 127, 128, 129, 1023, 1024, 1025, 8191, 8193, 1_300_003, 2_600_000]


@pytest.mark.parametrize("n", SIZES)
def test_tile_edges(n):
    G.load_library()
    rng = np.random.default_rng(n)
    deg = rng.integers(0, 3, size=n) if n > 3 else np.zeros(n, dtype=np.int64)
    off = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(deg, out=off[1:])
    first = rng.integers(0, max(1, n // 2), size=n)      # two neighbours at most, increasing
    src = np.repeat(np.arange(n), deg)
    nth = np.arange(off[-1]) - off[src]
    dst = (first[src] + nth * max(1, n // 2)).astype(np.int32)
    vl = rng.integers(0, 2, size=n).astype(np.int32)
    g = Graph(n, off, dst, np.zeros(off[-1], dtype=np.int32), vl, np.zeros((1, n), dtype=np.int32))
    dg = G.Graph(g)
    out = torch.full((n + 8,), -1, dtype=torch.int32, device="cuda")
    loops = np.bincount(src[src == dst], minlength=n)
    for label, need in ((-1, 0), (1, 1), (0, 2)):
        q = GFD([label] + [-1] * need, [(0, 1 + j, -1) for j in range(need)], [])
        want = np.flatnonzero(((vl == label) | (label < 0)) & (loops == 0) & (deg - loops >= need))
        for _ in range(2):
            got = G.node_candidates_noalloc(dg, q, 0, out.data_ptr(), out.numel())
            assert got == want.size
            np.testing.assert_array_equal(out[:got].cpu().numpy(), want)
