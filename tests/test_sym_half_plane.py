"""The symmetric pair kernel's half plane (CPU): with the sinks of an x-pencil and the sources of half a
plane, every ordered pair of cells of the (2R+1)^3 stencil is met exactly once in each direction."""
import os
import re

import pytest

HDR = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2110_11392_gb300", "csrc",
                   "nf_pair.cuh")


def half_table():
    text = re.search(r"c_half\[kHalfMax\]\[2\] = \{(.*?)\};", open(HDR).read(), re.S).group(1)
    return [tuple(int(v) for v in m) for m in re.findall(r"\{(-?\d+), (-?\d+)\}", text)]


@pytest.mark.parametrize("R", [1, 2, 3, 4])
def test_every_offset_once(R):
    nb = 1 + ((2 * R + 1) ** 2 - 1) // 2
    half = half_table()[:nb]
    assert half[0] == (0, 0) and [max(abs(b), abs(d)) for b, d in half] == sorted(max(abs(b), abs(d)) for b, d in half)
    assert {max(abs(b), abs(d)) for b, d in half[1:5]} == {1}  # the half first ring, then the others
    seen = []
    for c in range(-R, R + 1):          # sink cell, x offset from the pencil's centre
        for b, d in half:               # source cell, offset in the plane
            o = (-c, b, d)              # source minus sink
            if (b, d) != (0, 0):
                seen += [o, tuple(-v for v in o)]
            elif c < 0:                 # the centre cell acts both ways only on the sinks before it
                seen += [o, tuple(-v for v in o)]
            elif c == 0:
                seen += [o]             # a cell with itself: ordered pairs
    want = [(a, b, d) for a in range(-R, R + 1) for b in range(-R, R + 1) for d in range(-R, R + 1)]
    assert sorted(seen) == sorted(want)
