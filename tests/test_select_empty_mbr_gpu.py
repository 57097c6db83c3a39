"""Selection queries whose MBRs are empty (a low corner above the high one, as
an object without geometry has): they meet nothing, beside queries that do."""
import numpy as np
import pytest

from paper_2307_01716_gb300 import april as A
from tests.test_select_gpu import _check_grouping, ctx, run_select, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu

MAX, MIN = 2**31 - 1, -2**31
EMPTY = [(1 << 23, 0, 1 << 10, 1 << 24), (0, 1 << 23, 1 << 24, 1 << 10), (1 << 24, 1 << 24, 0, 0),
         (MAX, MAX, MIN, MIN), (MAX, 0, MIN, 1 << 24)]


@pytest.mark.parametrize("bits", [1, 4, 8])
def test_empty_mbrs_meet_nothing(torch_cuda, ctx, bits):  # noqa: F811
    rng = np.random.default_rng(bits)
    n, order = 500, 12
    lo = rng.integers(0, (1 << 24) - 70_000, (n, 2))
    mbr = np.concatenate([lo, lo + rng.integers(0, 70_000, (n, 2))], 1).astype(np.int32)
    cells = np.sort(rng.choice(1 << (2 * order), (n, 2), replace=False), 1)
    lists = [np.array([[a, b]]) for a, b in cells]
    none = np.zeros((0, 2))
    R = A.april_sets_from_lists(order, lists, [none] * n, mbr)
    whole = (0, 0, 1 << 24, 1 << 24)
    qm = np.array([EMPTY[0], whole, *EMPTY[1:], whole], dtype=np.int64).astype(np.int32)
    Q = A.april_sets_from_lists(order, lists[:len(qm)], [none] * len(qm), qm)
    dI = A.april_index_upload(A.april_index_build(R, bits))
    r, q, v, off = run_select(torch_cuda, ctx, dI, A.april_upload(R), A.april_upload(Q), len(qm), 2 * n)
    _check_grouping(r, q, off, len(qm))
    assert np.array_equal(np.diff(off.astype(np.int64)), [0, n, 0, 0, 0, 0, n])
    assert np.array_equal(np.sort(r[:n]), np.arange(n)) and np.array_equal(np.sort(r[n:]), np.arange(n))
    want, _ = A.april_host_filter(R, Q, r, q)
    assert np.array_equal(v, want)
