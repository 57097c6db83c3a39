"""The filter variants' window waits that run out (GPU only): with the
single lanes off, april_filter_pairs_ex joins by warps and, above a threshold,
by warps or CTAs; the diagnostic wait limit 0 makes each wait give up, the
pairs held read as errors, april_sync_status reports the timeout, and the next
call is right."""
import numpy as np
import pytest

from paper_2307_01716_gb300 import april as A
from tests.test_timeout_gpu import _run, setup  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threshold,window", [(0xFFFFFFFF, 128), (2048, 64), (2048, 256)])
@pytest.mark.parametrize("predicate", [A.PREDICATE_INTERSECTS, A.PREDICATE_WITHIN])
def test_variant_waits_run_out(setup, threshold, window, predicate):  # noqa: F811
    torch, w, dR, dS, d_r, d_s, _ = setup
    n = len(w.pr)
    ctx = A.Context(0)
    t = ctx.get_tune()
    t.triage_off, t.cta_threshold, t.cta_window = 1, threshold, window
    ctx.set_tune(t)
    scratch = torch.empty(ctx.scratch_bytes(A.MODE_BATCHED, n), dtype=torch.uint8, device="cuda")
    want = torch.full((n,), 0xEE, dtype=torch.uint8, device="cuda")
    A.Context(0).april_filter_pairs_ex(dR, dS, d_r, d_s, n, want, predicate, scratch)  # by single lanes
    torch.cuda.synchronize()
    _run(torch, ctx, lambda out: ctx.april_filter_pairs_ex(dR, dS, d_r, d_s, n, out, predicate, scratch), n)
    out = torch.full((n,), 0xEE, dtype=torch.uint8, device="cuda")
    ctx.april_filter_pairs_ex(dR, dS, d_r, d_s, n, out, predicate, scratch)
    ctx.april_sync_status()
    assert np.array_equal(out.cpu().numpy(), want.cpu().numpy())
