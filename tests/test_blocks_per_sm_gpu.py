"""april_tune.blocks_per_sm in the default shape: the grid of the lane kernels
follows it (a call at one CTA per SM takes longer than at as many as fit,
through april_filter_pairs and the host entry point), the verdicts do not."""
import numpy as np
import pytest

from tests import _data
from paper_2307_01716_gb300 import april as A

pytestmark = pytest.mark.gpu


def test_lane_grids_follow_blocks_per_sm():
    torch = pytest.importorskip("torch")
    w = _data.workload(3, 0.01)
    g = A.global_grid(w.order)
    R, S = A.april_build_sets(w.R.xy, w.R.off, g), A.april_build_sets(w.S.xy, w.S.off, g)
    want, _ = A.april_host_filter(R, S, w.pr, w.ps)
    rep = -(-800_000 // len(w.pr))
    pr, ps, want = (np.tile(v, rep) for v in (w.pr, w.ps, want))
    n = len(pr)
    dR, dS = A.april_upload(R), A.april_upload(S)
    h_r, h_s = (torch.from_numpy(v.view(np.int32)).pin_memory() for v in (pr, ps))
    d_r, d_s = h_r.cuda(), h_s.cuda()
    ctx = A.Context(0)
    out = torch.empty(n, dtype=torch.uint8, device="cuda")
    h_v = torch.empty(n, dtype=torch.uint8).pin_memory()
    scratch = torch.empty(ctx.scratch_bytes(A.MODE_BATCHED, n), dtype=torch.uint8, device="cuda")
    work = torch.empty(ctx.host_work_bytes(A.MODE_BATCHED, n), dtype=torch.uint8, device="cuda")

    def run(blocks, call, verdicts):
        t = ctx.get_tune()
        t.blocks_per_sm = blocks
        ctx.set_tune(t)
        ms = []
        for _ in range(8):
            verdicts.fill_(0xEE)
            torch.cuda.synchronize()
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            call()
            b.record()
            torch.cuda.synchronize()
            ms.append(a.elapsed_time(b))
        ctx.april_sync_status()
        assert np.array_equal(verdicts.cpu().numpy(), want)
        return float(np.median(ms[2:]))

    def batched():
        ctx.april_filter_pairs(dR, dS, d_r, d_s, n, out, A.MODE_BATCHED, scratch)

    def host():
        ctx.april_filter_pairs_host(dR, dS, h_r, h_s, n, h_v, A.MODE_BATCHED, work)

    # the kernels hide latency by warps: a fifth of them takes well over twice as long
    # (the host entry point's copies take part of a call, so less of it)
    for call, verdicts, factor in ((batched, out, 1.5), (host, h_v, 1.3)):
        most, one, again = (run(b, call, verdicts) for b in (0, 1, 0))
        assert one > factor * max(most, again), (most, one, again)
