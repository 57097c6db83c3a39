"""The autotuner's candidates: the single lanes are one of them, not one per
group shape that they do not read, and the lane groups without a threshold
are candidates of their own."""
import numpy as np
import pytest

from tests import _data
from paper_2307_01716_gb300 import april as A

pytestmark = pytest.mark.gpu


def test_candidates_differ():
    torch = pytest.importorskip("torch")
    w = _data.workload(3, 0.01)
    g = A.global_grid(w.order)
    R, S = A.april_build_sets(w.R.xy, w.R.off, g), A.april_build_sets(w.S.xy, w.S.off, g)
    dR, dS = A.april_upload(R), A.april_upload(S)
    n = len(w.pr)
    d_r, d_s = (torch.from_numpy(v.view(np.int32)).cuda() for v in (w.pr, w.ps))
    ctx = A.Context(0)
    d = ctx.get_tune()
    out = torch.empty(n, dtype=torch.uint8, device="cuda")
    scratch = torch.empty(ctx.scratch_bytes(A.MODE_BATCHED, n), dtype=torch.uint8, device="cuda")
    slow = A.april_tune(2048, 32, 32, 2048, 1)  # whole warps and CTAs, at one CTA per SM
    ctx.set_tune(slow)
    t = ctx.april_autotune(dR, dS, d_r, d_s, n, out, scratch)
    captures, launches = ctx.april_ctx_graph_stats()
    # the context's own tuning; per join order the lanes, four thresholds x ten shapes x three scopes, ten shapes
    candidates = 1 + 2 * (1 + 4 * 10 * 3 + 10)
    assert (captures, launches) == (candidates, 4 * candidates)
    if t.cta_threshold == d.cta_threshold and t.group_lanes < 32 and not t.triage_off:  # the lanes
        assert (t.group_lanes, t.group_window) == (d.group_lanes, d.group_window)
    want, _ = A.april_host_filter(R, S, w.pr, w.ps)
    out.fill_(0xEE)
    ctx.april_filter_pairs(dR, dS, d_r, d_s, n, out, A.MODE_BATCHED, scratch)
    ctx.april_sync_status()
    assert np.array_equal(out.cpu().numpy(), want)
