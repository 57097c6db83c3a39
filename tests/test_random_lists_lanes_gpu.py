"""The filter variants in the default shape (single lanes, and 8 to 32 lanes
per pair of a call of few) on the random and adversarial lists, against the
host, in both join orders."""
import numpy as np
import pytest

from paper_2307_01716_gb300 import april as A
from tests.test_random_lists_gpu import _run, ctx, data, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("join_order", [0, 1])
@pytest.mark.parametrize("which", ["within", "within S", "intersects", "coarser S", "coarser R"])
def test_lane_variants_equal_host(torch_cuda, ctx, data, which, join_order):  # noqa: F811
    R, S, S14, pr, ps = data
    X, Y, pred = {"within": (R, S, A.PREDICATE_WITHIN), "within S": (S, R, A.PREDICATE_WITHIN),
                  "intersects": (R, S, A.PREDICATE_INTERSECTS), "coarser S": (R, S14, A.PREDICATE_INTERSECTS),
                  "coarser R": (S14, R, A.PREDICATE_INTERSECTS)}[which]
    if which == "within S":
        pr, ps = ps, pr
    want, _ = A.april_host_filter_ex(X, Y, pr, ps, pred)
    dX, dY = A.april_upload(X), A.april_upload(Y)
    saved = ctx.get_tune()
    t = ctx.get_tune()
    t.join_order = join_order
    ctx.set_tune(t)

    def fn(d_r, d_s, out, n):
        scratch = torch_cuda.empty(ctx.scratch_bytes(A.MODE_BATCHED, n), dtype=torch_cuda.uint8, device="cuda")
        ctx.april_filter_pairs_ex(dX, dY, d_r, d_s, n, out, pred, scratch)

    try:
        # 32, 16 and 8 lanes a pair, more pairs than the first ones of every resident warp, a lane a pair
        for n in (900, 9_000, 20_000, 40_000, len(pr)):
            got = _run(torch_cuda, ctx, dX, dY, pr[:n], ps[:n], fn)
            bad = np.flatnonzero(got != want[:n])
            assert len(bad) == 0, (n, len(bad), bad[:10])
    finally:
        ctx.set_tune(saved)
