"""Selection with a warp per query (very many queries) and with a CTA per
query: the same pairs in the same order, equal to the MBR step by brute force,
for queries of no, one and many bucket rows."""
import numpy as np
import pytest

from paper_2307_01716_gb300 import april as A
from tests.test_select_gpu import _check_grouping, ctx, run_select, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu

L = 1 << 24


def _sets(rng, n, sizes):
    lo = rng.integers(0, L, (n, 2))
    w = rng.choice(sizes, n)[:, None] * rng.random((n, 2))
    mbr = np.concatenate([lo, np.minimum(lo + w, L)], 1).astype(np.int64)
    cells = np.sort(rng.integers(0, 1 << 24, (n, 1)), 1)
    lists = list(np.concatenate([cells, cells + 1], 1)[:, None])
    return A.april_sets_from_lists(12, lists, [np.zeros((0, 2))] * n, mbr.astype(np.int32)), mbr


@pytest.mark.parametrize("bits", [1, 6, 8])
def test_warp_and_cta_queries_agree(torch_cuda, ctx, bits):  # noqa: F811
    rng = np.random.default_rng(bits)
    n, nq = 400, 30_000
    R, rm = _sets(rng, n, [1e3, 1e5, 3e6])
    Q, qm = _sets(rng, nq, [1e3, 3e5, 1e7])
    dR = A.april_upload(R)
    dI = A.april_index_upload(A.april_index_build(R, bits))
    meet = (rm[None, :, 0] <= qm[:, None, 2]) & (qm[:, None, 0] <= rm[None, :, 2]) & \
        (rm[None, :, 1] <= qm[:, None, 3]) & (qm[:, None, 1] <= rm[None, :, 3])
    want_q, want_r = np.nonzero(meet)
    r, q, v, off = run_select(torch_cuda, ctx, dI, dR, A.april_upload(Q), nq, len(want_r) + 1)
    _check_grouping(r, q, off, nq)
    by = np.lexsort((r, q))
    assert np.array_equal(r[by], want_r) and np.array_equal(q[by], want_q)
    hv, _ = A.april_host_filter(R, Q, r, q)
    assert np.array_equal(v, hv)
    # few queries at a time: a CTA each
    for a in (0, 12_345, nq - 2_000):
        lists = [[Q.list(i, w) for i in range(a, a + 2_000)] for w in (0, 1)]
        P = A.april_sets_from_lists(12, *lists, qm[a:a + 2_000].astype(np.int32))
        r2, q2, v2, _ = run_select(torch_cuda, ctx, dI, dR, A.april_upload(P), 2_000, int(off[a + 2_000] - off[a]))
        sl = slice(int(off[a]), int(off[a + 2_000]))
        assert np.array_equal(r2, r[sl]) and np.array_equal(q2 + a, q[sl]) and np.array_equal(v2, v[sl])
