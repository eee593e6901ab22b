"""Integration at scan sizes that take each tile of returns (4, 8, 12, 16) for
each class of cube: several CTAs per SM, two, one. Map and caller's box against
the oracle, as in test_gpu_box_tiles.py, with a last tile that is not full."""
import pytest

import test_gpu_box_tiles as tiles

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("radius,n", [(1, 6001), (2, 9001), (2, 14003)] +
                         [(3, n) for n in (3001, 6003, 8005, 12007)] +
                         [(4, n) for n in (1001, 2003, 2805, 4007)] +
                         [(5, n) for n in (1003, 2001, 3007)] +
                         [(7, n) for n in (501, 1005, 1803, 2207)])
def test_each_tile(radius, n):
    tiles.test_box_tiles(radius=radius, n=n)
