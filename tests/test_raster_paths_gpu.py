"""GPU construction at the sizes where a polygon's path changes (a warp's
window of 64 x 64 cells, a CTA's of 256 x 256, tiles, sorted cells): lists
equal to the host builder's, list for list."""
import numpy as np
import pytest

from paper_2307_01716_gb300 import april as A
from tests.test_build_device_gpu import _check_equal_host, _pack, _rect, ctx, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu

WIDTHS = [1, 2, 7, 8, 9, 63, 64, 65, 127, 129, 255, 256, 257, 511, 513, 770]


def _star(rng, cx, cy, rad, n):
    a = np.sort(rng.uniform(0, 2 * np.pi, n))
    r = rad * rng.uniform(0.3, 1.0, n)
    p = np.stack([cx + r * np.cos(a), cy + r * np.sin(a)], 1).round().astype(np.int64)
    return np.concatenate([p, p[-1:]])  # a vertex twice: an edge that is a point


def _polygons(order, log2_cell, ox, oy, seed):
    rng = np.random.default_rng(seed)
    h, side = 1 << log2_cell, 1 << order
    out = []
    for w in WIDTHS:
        if w > side:
            continue
        x, y = (int(v) for v in rng.integers(0, side - w + 1, 2))
        x0, y0 = ox + x * h, oy + y * h
        out.append(_rect(x0, y0, x0 + w * h, y0 + w * h))                       # along grid lines
        out.append(_rect(x0, y0, x0 + w * h, y0 + max(h // 2, 1)))              # one cell high
        out.append(_rect(x0 + h // 3, y0, x0 + h // 3 + max(h // 4, 1), y0 + w * h))  # one wide
        for n in (5, 40):
            out.append(_star(rng, x0 + w * h / 2, y0 + w * h / 2, max(w * h / 2, 2 * h), n))
    # outlines that cross the grid in a few cells and hold most of it: sorted where the grid has many tiles
    g = side * h
    for c in (1, 3, 40):
        k = min(c, side - 1) * h + h // 2
        out.append(np.array([[ox - 3 * h, oy - 3 * h], [ox + g + 3 * h, oy - 3 * h], [ox + g + 3 * h, oy + g - k],
                             [ox + g - k, oy + g + 3 * h], [ox - 3 * h, oy + g + 3 * h]], dtype=np.int64))
    far = (1 << 26) - g - 32  # about as wide as the builder takes
    out.append(np.array([[ox - far, oy - 5], [ox + g // 2, oy + g // 3 + 1], [ox - 7, oy + g + 5]], dtype=np.int64))
    return out


@pytest.mark.parametrize("order,log2_cell,ox,oy", [(1, 6, 0, 0), (3, 4, 0, 0), (6, 1, 77, -13), (8, 3, 1000, 3000),
                                                   (9, 5, 0, 0), (11, 2, -5000, 12345), (13, 2, 1 << 20, 1 << 19),
                                                   (16, 8, 0, 0)])
def test_paths_equal_host(torch_cuda, ctx, order, log2_cell, ox, oy):  # noqa: F811
    xy, off = _pack(_polygons(order, log2_cell, ox, oy, order))
    _check_equal_host(torch_cuda, ctx, xy, off, A.april_grid(ox, oy, log2_cell, order))
