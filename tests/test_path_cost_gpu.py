"""GPU construction of outlines with many vertices over many tiles: the time
follows the touched cells, not vertices times tiles, and the lists equal the
host builder's whichever path the polygons take."""
import numpy as np
import pytest

from paper_2307_01716_gb300 import april as A
from tests.test_build_device_gpu import _check_equal_host, _device_polys, _pack, ctx, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def _outlines(rng, count, verts, radius, jag=0.0):
    """Smooth closed curves of about `radius` cells of 2^8 (order 16), with `jag` of it added at random."""
    th = (np.arange(verts) + 0.5) / verts * 2 * np.pi
    polys = []
    for _ in range(count):
        r = 1 + sum(0.5 / k * np.sin(k * th + rng.uniform(0, 6.28)) for k in (2, 3, 5, 9, 17, 33, 65, 129))
        r = np.maximum(r, 0.1) * (1 + jag * rng.uniform(-0.5, 0.5, verts)) * radius * 128
        c = rng.uniform(1.3, (1 << 16) / radius - 1.3, 2) * radius * 256
        polys.append((c + r[:, None] * np.stack([np.cos(th), np.sin(th)], 1)).round().clip(0, 1 << 24))
    return _pack([p.astype(np.int64) for p in polys])


def _ms(torch, ctx, xy, off, grd):  # noqa: F811
    d = _device_polys(torch, xy, off)
    dev, info = ctx.april_build_sets_device(*d, grd)
    work = torch.empty(int(info.work_bytes), dtype=torch.uint8, device="cuda")
    ms = []
    for _ in range(5):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        torch.cuda.synchronize()
        a.record()
        ctx.april_build_sets_device(*d, grd, work, dev.buf)
        b.record()
        torch.cuda.synchronize()
        ms.append(a.elapsed_time(b))
    return min(ms), info.touched_cells


def test_time_follows_cells(torch_cuda, ctx):  # noqa: F811
    g = A.global_grid(16)
    rng = np.random.default_rng(1)
    few, few_cells = _ms(torch_cuda, ctx, *_outlines(rng, 100, 1_000, 4000), g)
    many, cells = _ms(torch_cuda, ctx, *_outlines(rng, 100, 100_000, 4000), g)
    # the same windows and tiles; the cells grow five times, vertices x tiles a hundred times
    assert many / few < cells / few_cells, (few, many, few_cells, cells)


@pytest.mark.parametrize("count,verts,radius,jag", [(3, 50_000, 2000, 0.0), (60, 300, 6000, 0.0), (60, 300, 6000, 0.4),
                                                    (300, 64, 2500, 0.1), (2, 400, 20000, 0.2)])
def test_both_sides_equal_host(torch_cuda, ctx, count, verts, radius, jag):  # noqa: F811
    xy, off = _outlines(np.random.default_rng(verts), count, verts, radius, jag)
    _check_equal_host(torch_cuda, ctx, xy, off, A.global_grid(16))
