"""The batched pipeline's captured graph is replayed only for the arguments it
holds: a set uploaded into the buffer of another, with the same objects and
interval slots but another number of compressed blocks (its gap stream lies
elsewhere in the image), gets its own verdicts."""
import ctypes

import numpy as np
import pytest

from paper_2307_01716_gb300 import april as A

pytestmark = pytest.mark.gpu


def _sets(rng, lengths):
    lists = []
    for n in lengths:
        st = 2 * np.sort(rng.choice(300, n, replace=False)).astype(np.uint64)
        lists.append(np.stack([st, st + 1], 1))
    R = A.april_sets_from_lists(8, lists, [v[::5] for v in lists])
    R.compress()
    return R


def test_second_upload_into_one_buffer():
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(3)
    n = 64
    sets = [_sets(rng, [16, 16] * (n // 2)), _sets(rng, [18, 14] * (n // 2))]
    S = _sets(rng, rng.integers(1, 30, n))
    infos = [R.info() for R in sets]
    assert infos[0].iv_slots == infos[1].iv_slots and infos[0].device_bytes != infos[1].device_bytes
    dS = A.april_upload(S)
    g = np.indices((n, n)).reshape(2, -1).astype(np.uint32)
    pr, ps = np.ascontiguousarray(g[0]), np.ascontiguousarray(g[1])
    k = len(pr)
    d_r, d_s = (torch.from_numpy(v.view(np.int32)).cuda() for v in (pr, ps))
    out = torch.empty(k, dtype=torch.uint8, device="cuda")
    ctx = A.Context(0)
    scratch = torch.empty(ctx.scratch_bytes(A.MODE_BATCHED_PACKED, k), dtype=torch.uint8, device="cuda")
    buf = torch.zeros(1 << 20, dtype=torch.uint8, device="cuda")  # far more than either image
    for R in sets + sets[:1]:
        dR = A.DevSets(A.april_dev_sets(), buf)
        A.check(A.load().april_upload(R.handle, buf.data_ptr(), buf.numel(),
                                      torch.cuda.current_stream().cuda_stream, ctypes.byref(dR.c)))
        out.fill_(0xEE)
        ctx.april_filter_pairs(dR, dS, d_r, d_s, k, out, A.MODE_BATCHED_PACKED, scratch)
        ctx.april_sync_status()
        want, _ = A.april_host_filter(R, S, pr, ps)
        assert np.array_equal(out.cpu().numpy(), want)
