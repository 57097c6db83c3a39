"""Compressed sets whose block table is very large: verdicts do not depend on
where in the table a list's blocks lie, below, across and above block 2^28,
from which on 16 slots a block no longer fit 32 bits.  A small set stands in
for the large one: its block numbers are raised by a constant and its table's
address lowered to match, so every access stays in the small table."""
import ctypes

import numpy as np
import pytest

from paper_2307_01716_gb300 import april as A

pytestmark = pytest.mark.gpu


def _raised(torch, dev, n, by):
    """A copy of the device sets whose block numbers lie `by` higher."""
    c = A.april_dev_sets()
    ctypes.memmove(ctypes.byref(c), ctypes.byref(dev.c), ctypes.sizeof(c))
    base = dev.buf.data_ptr()
    pdesc = dev.buf[dev.c.pdesc - base:dev.c.pdesc - base + 16 * n].clone().view(torch.int32).view(n, 4)
    pdesc[:, 0::2] += by
    torch.cuda.synchronize()
    c.pdesc, c.anchors = pdesc.data_ptr(), dev.c.anchors - 8 * by
    out = A.DevSets.__new__(A.DevSets)
    out.__dict__.update(dev.__dict__)
    out.c, out.kept = c, pdesc
    return out


@pytest.mark.parametrize("by", [0, 1 << 27, (1 << 28) - 64, (1 << 28) + 96])
def test_block_numbers_around_2_28(by):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(28)

    def lists():
        a, f = [], []
        for n in (0, 1, 15, 16, 17, 40, 200, 200, 333, 1000):
            p = np.unique(rng.integers(0, 1 << 16, 3 * n + 8))[:2 * n] + int(rng.integers(0, 1 << 16))
            iv = p.reshape(-1, 2).astype(np.uint64)
            keep = np.ones(len(iv), bool)
            keep[1:] = iv[1:, 0] > iv[:-1, 1]
            a.append(iv[keep])
            f.append(a[-1][rng.random(len(a[-1])) < 0.1])
        return A.april_sets_from_lists(16, a, f), len(a)

    (R, n), (S, m) = lists(), lists()
    g = np.indices((n, m)).reshape(2, -1).astype(np.uint32)
    pr, ps = np.ascontiguousarray(g[0]), np.ascontiguousarray(g[1])
    want, _ = A.april_host_filter(R, S, pr, ps)
    assert (np.bincount(want, minlength=3) > 5).all()
    R.compress(), S.compress()
    dR, dS = _raised(torch, A.april_upload(R), n, by), _raised(torch, A.april_upload(S), m, by)
    ctx = A.Context(0)
    for rep in (1, 600):  # few pairs, and more than eight for every resident warp
        k = len(pr) * rep
        d_r, d_s = (torch.from_numpy(np.tile(v, rep).view(np.int32)).cuda() for v in (pr, ps))
        out = torch.full((k,), 0xEE, dtype=torch.uint8, device="cuda")
        scratch = torch.empty(ctx.scratch_bytes(A.MODE_BATCHED_PACKED, k), dtype=torch.uint8, device="cuda")
        ctx.april_filter_pairs(dR, dS, d_r, d_s, k, out, A.MODE_BATCHED_PACKED, scratch)
        ctx.april_sync_status()
        assert np.array_equal(out.cpu().numpy(), np.tile(want, rep))
        h = [t.cpu().pin_memory() if rep == 1 else t.cpu() for t in (d_r, d_s)]
        h_v = torch.full((k,), 0xEE, dtype=torch.uint8)
        work = torch.empty(ctx.host_work_bytes(A.MODE_BATCHED_PACKED, k), dtype=torch.uint8, device="cuda")
        ctx.april_filter_pairs_host(dR, dS, *h, k, h_v, A.MODE_BATCHED_PACKED, work)
        assert np.array_equal(h_v.numpy(), np.tile(want, rep))
