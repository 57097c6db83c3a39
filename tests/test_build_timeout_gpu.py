"""The bounded wait of the GPU construction (GPU only): a tile of a large
polygon waits for the sums of the tiles before it.  With the diagnostic wait
limit at 0 every such wait gives up at once, with no fault: the polygons
concerned get empty lists, the others theirs, april_sync_status reports the
timeout, and the next build at the default limit is right again."""
import numpy as np
import pytest

from paper_2307_01716_gb300 import april as A
from tests.test_build_device_gpu import (_check_equal_host, _device_polys, _pack, _read_lists, _rect, ctx,  # noqa: F401
                                         torch_cuda)

pytestmark = pytest.mark.gpu


def test_build_wait_runs_out(torch_cuda, ctx):  # noqa: F811
    order, log2_cell = 12, 4
    h = 1 << log2_cell
    # windows of 40, 200, 600, 1,000 and 3,000 cells: the last three are tiled
    polys = [_rect(5 * h + 3, 7 * h, (5 + w) * h, (7 + w) * h - 5) for w in (40, 200, 600, 1000, 3000)] * 3
    tiled = [w > 256 for w in (40, 200, 600, 1000, 3000)] * 3
    xy, off = _pack(polys)
    g = A.april_grid(0, 0, log2_cell, order)
    H, dev, _ = _check_equal_host(torch_cuda, ctx, xy, off, g)
    try:
        A.april_debug_set_wait_limit(0)
        dev, _ = ctx.april_build_sets_device(*_device_polys(torch_cuda, xy, off), g)
        torch_cuda.cuda.synchronize()
    finally:
        A.april_debug_set_wait_limit(A.WAIT_LIMIT_DEFAULT)
    with pytest.raises(A.AprilError) as e:
        ctx.april_sync_status()
    assert e.value.status == -5
    lists, mbr = _read_lists(dev, len(polys))
    for p, t in enumerate(tiled):
        if t:
            assert len(lists[p][0]) == 0 and len(lists[p][1]) == 0, p
        else:
            assert np.array_equal(lists[p][0], H.list(p, 0)) and np.array_equal(lists[p][1], H.list(p, 1)), p
    assert np.array_equal(mbr, H.mbrs())
    _check_equal_host(torch_cuda, ctx, xy, off, g)
    ctx.april_sync_status()
