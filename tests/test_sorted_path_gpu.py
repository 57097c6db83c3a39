"""GPU construction of many polygons that are built from their sorted cells
(outlines that meet few cells of a window of many tiles), spread over several
blocks of polygon records and mixed with small ones: one sort orders the keys
of all of them by polygon, so every polygon's range has to lie in polygon
order.  Lists equal to the host builder's, list for list."""
import numpy as np
import pytest

from paper_2307_01716_gb300 import april as A
from tests.test_build_device_gpu import _check_equal_host, _pack, _rect, ctx, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 33, 2049, 6200])
def test_sorted_ranges_follow_polygon_order(torch_cuda, ctx, n):  # noqa: F811
    order, log2_cell = 12, 4
    h, g = 1 << log2_cell, 1 << (order + log2_cell)
    rng = np.random.default_rng(n)
    polys = []
    for p in range(n):
        if p % 3 == 2:
            x, y = (int(v) for v in rng.integers(0, g - 40 * h, 2))
            w = int(rng.integers(1, 40 * h))
            polys.append(_rect(x, y, x + w, y + w))
        else:  # the grid less a corner: from a few cells up to a few hundred of 2^24
            k = int(rng.integers(1, 120)) * h + int(rng.integers(0, h))
            polys.append(np.array([[-3 * h, -3 * h], [g + 3 * h, -3 * h], [g + 3 * h, g - k], [g - k, g + 3 * h],
                                   [-3 * h, g + 3 * h]], dtype=np.int64))
    xy, off = _pack(polys)
    _check_equal_host(torch_cuda, ctx, xy, off, A.april_grid(0, 0, log2_cell, order))
