"""Memory of thin specimens, whose cell grid is mostly empty (its margin follows
the longest edge): two lists, the atoms' arrays and 8 bytes per cell of about
the list radius cubed."""
import math

import pytest


@pytest.mark.parametrize("shape,prec", [((1000, 1, 3), 0), ((400, 3, 3), 0), ((80, 3, 3), 1)])
def test_cells_of_thin_specimens_are_not_divided(shape, prec):
    import paper_2603_07321_gb300 as P
    P.build()
    n = 4 * shape[0] * shape[1] * shape[2]
    p = P.default_params(precision=prec)
    edge = 2 * 4.05 + p.skin
    longest = 4.05 * max(shape)
    cells = math.prod((4.05 * s + 0.5 * longest + 4 * edge) / edge + 2 for s in shape)
    capacity = 1.6 * 4 / 3 * math.pi * edge**3 * 4 / 4.05**3 + 48
    lists = 2 * 4 * n * (capacity + 16 * 12 + 4)
    got = P.pta_footprint_bytes(P.make_specimen(shape), p)
    assert got < 8 * cells + lists + 1200 * n + 100e3
