"""GFDs held in other containers than lists, tuples and arrays: the binding takes and
refuses what its conversion by numpy does, with the same image."""
from array import array

import pytest

from synth.gfds import GFD, Literal

import paper_2608_02321_gb300 as G
from test_binding_marshalling import _image, _Slow

ONE = [Literal.const(0, 0, 1)]

REFUSED = [
    lambda: GFD(b"\1\0\0\0\2\0\0\0", []),
    lambda: GFD({1, 2}, []),
    lambda: GFD({1: 0}, []),
    lambda: GFD((x for x in (1, 2)), []),
    lambda: GFD([0, 1], (e for e in [(0, 1, -1)])),
    lambda: GFD([0, 1], {(0, 1, -1)}),
    lambda: GFD([0, 1], {(0, 1, -1): 1}),
    lambda: GFD([0, 1], [{0, 1, 2}]),
    lambda: GFD([0, 1], [b"\0\1\2"]),
    lambda: GFD([0], [], iter(ONE)),
    lambda: GFD([0], [], [], (q for q in ONE)),
]
TAKEN = [
    lambda: GFD(bytearray(8), []),              # eight labels, not two
    lambda: GFD(range(3), [(0, 1, -1)]),
    lambda: GFD(array("q", [4, 5]), []),
    lambda: GFD([0], [], {ONE[0]: 1}, set(ONE)),
]


@pytest.mark.parametrize("i", range(len(REFUSED)))
def test_refused(i):
    with pytest.raises(Exception) as want:
        _Slow(REFUSED[i]())
    with pytest.raises(type(want.value)):
        G._GfdBuf(REFUSED[i]())


@pytest.mark.parametrize("i", range(len(TAKEN)))
def test_taken(i):
    assert _image(G._GfdBuf(TAKEN[i]())) == _image(_Slow(TAKEN[i]()))
