"""The binding's two ways to lay out a GFD (packed arrays for plain whole numbers,
numpy and ctypes for everything else) give the same image."""
import ctypes as C

import numpy as np
import pytest

from synth.gfds import GFD, Literal

import paper_2608_02321_gb300 as G


def _image(buf):
    s = buf.s

    def ints(p, n):
        return list((C.c_int32 * n).from_address(p)) if n else []
    return (s.k, ints(s.node_label, s.k), s.m, ints(s.esrc, s.m), ints(s.edst, s.m), ints(s.elabel, s.m),
            s.nx, ints(s.X, 6 * s.nx), s.ny, ints(s.Y, 6 * s.ny), s.y_false)


class _Slow(G._GfdBuf):
    def __init__(self, gfd):
        self._convert(gfd)


LITS = [Literal.const(0, 1, 7), Literal.var(1, 2, 0, 3)]
CASES = [
    GFD([0, -1, 2], [(0, 1, -1), (1, 2, 3)], LITS, LITS[:1]),
    GFD([5], [], [], [], True),
    GFD(np.array([1, 2]), np.array([[0, 1, 4]]), [], LITS),               # arrays
    GFD(np.array([1, 2], dtype=np.uint8), [np.array([0, 1, 4])], [], []),
    GFD((3, 4), ((0, 1, np.int64(2)),), (), ()),
    GFD([1.0, 2.0], [(0, 1, 2)], [], []),                                  # converted by numpy
    GFD([1, 2], [0, 1, 2, 1, 0, 3], [], []),                               # flat edges
    GFD([1, 2], [(0, 1, True)], [Literal.const(0, 0, 2 ** 31 + 5)], []),   # wraps, as ctypes does
]


@pytest.mark.parametrize("i", range(len(CASES)))
def test_same_image(i):
    assert _image(G._GfdBuf(CASES[i])) == _image(_Slow(CASES[i]))


@pytest.mark.parametrize("bad", [GFD([0, 1], [(0, 1)]), GFD([2 ** 40], []), GFD(["a"], []), GFD([0], [(0, 0, None)])])
def test_same_refusal(bad):
    with pytest.raises(Exception) as want:
        _Slow(bad)
    with pytest.raises(type(want.value)):
        G._GfdBuf(bad)
