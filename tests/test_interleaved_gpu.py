"""Large calls over finely interleaved lists, whose joins use up their rounds
in a single lane and go on in merge windows: verdicts equal the host's through
every entry point, at whichever of its joins a pair is handed over, and a call
does not take many times as long as with the windows alone."""
import numpy as np
import pytest

from paper_2307_01716_gb300 import april as A

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _sets(rng, side, order=16):
    """Lists of single cells 8 i + 3 side; some cells of the other side's added here and there; F none, a few or most."""
    a, f = [], []
    for n in (1, 7, 23, 24, 25, 60, 200, 201, 500, 1500, 40, 90, 333, 700):
        for extra in (0, 1, 30):
            i = np.sort(rng.choice(max(2 * n, 3), n, replace=False)) if extra == 30 else np.arange(n)
            x = 8 * i + 100 + 3 * side
            # cells of the other side, late in the list
            y = rng.choice(np.arange(max(2 * n // 3, 0), 2 * n + 1), min(extra, n)) * 8 + 100 + 3 * (1 - side)
            x = np.unique(np.concatenate([x, y])).astype(np.uint64)
            iv = np.stack([x, x + 1], 1)
            a.append(iv)
            f.append(iv[rng.random(len(iv)) < rng.choice([0.0, 0.05, 0.6])])
    return a, f, A.april_sets_from_lists(order, a, f)


def _ctx(off):
    ctx = A.Context(0)
    t = ctx.get_tune()
    t.triage_off = off
    ctx.set_tune(t)
    return ctx


@pytest.fixture(scope="module")
def data():
    rng = np.random.default_rng(16)
    (_, _, R), (sa, sf, S) = _sets(rng, 0), _sets(rng, 1)
    S14 = A.april_sets_from_lists(14, [np.stack([u := np.unique(v[:, 0] >> np.uint64(4)), u + np.uint64(1)], 1)
                                       for v in sa],
                                  [np.stack([u := np.unique(v[:, 0] >> np.uint64(4)), u + np.uint64(1)], 1) for v in sf])
    n = 200_000
    pr, ps = (rng.integers(0, len(sa), n).astype(np.uint32) for _ in range(2))
    return R, S, S14, pr, ps


def test_batched_and_host(torch_cuda, data):
    torch = torch_cuda
    R, S, _, pr, ps = data
    n = len(pr)
    want, _ = A.april_host_filter(R, S, pr, ps)
    assert (np.bincount(want, minlength=3) > 1000).all()
    R.compress(), S.compress()
    dR, dS = A.april_upload(R), A.april_upload(S)
    h_r, h_s = (torch.from_numpy(v.view(np.int32)) for v in (pr, ps))
    d_r, d_s = h_r.cuda(), h_s.cuda()
    for jo in (0, 1):
        for lanes, window, escalate in ((4, 32, 0), (8, 16, 0), (16, 64, 2)):
            ctx = A.Context(0)
            t = ctx.get_tune()
            t.join_order, t.group_lanes, t.group_window, t.escalate_windows = jo, lanes, window, escalate
            ctx.set_tune(t)
            for mode in (A.MODE_BATCHED, A.MODE_BATCHED_PACKED):
                out = torch.full((n,), 0xEE, dtype=torch.uint8, device="cuda")
                scratch = torch.empty(ctx.scratch_bytes(mode, n), dtype=torch.uint8, device="cuda")
                ctx.april_filter_pairs(dR, dS, d_r, d_s, n, out, mode, scratch)
                ctx.april_sync_status()
                assert np.array_equal(out.cpu().numpy(), want), (jo, lanes, mode)
                work = torch.empty(ctx.host_work_bytes(mode, n), dtype=torch.uint8, device="cuda")
                for pin in (False, True):
                    p = [v.pin_memory() if pin else v for v in (h_r, h_s)]
                    h_v = torch.full((n,), 0xEE, dtype=torch.uint8)
                    ctx.april_filter_pairs_host(dR, dS, *p, n, h_v, mode, work)
                    assert np.array_equal(h_v.numpy(), want), (jo, lanes, mode, pin)
    out = torch.full((n,), 0xEE, dtype=torch.uint8, device="cuda")
    A.april_filter_pairs_noalloc(dR, dS, d_r, d_s, n, out)
    A.april_noalloc_sync_status()
    assert np.array_equal(out.cpu().numpy(), want)


@pytest.mark.parametrize("which", ["within", "within S", "intersects", "coarser S", "coarser R"])
def test_variants(torch_cuda, data, which):
    torch = torch_cuda
    R, S, S14, pr, ps = data
    X, Y, pred = {"within": (R, S, 1), "within S": (S, R, 1), "intersects": (R, S, 0), "coarser S": (R, S14, 0),
                  "coarser R": (S14, R, 0)}[which]
    n = len(pr)
    want, _ = A.april_host_filter_ex(X, Y, pr, ps, pred)
    dX, dY = A.april_upload(X), A.april_upload(Y)
    d_r, d_s = (torch.from_numpy(v.view(np.int32)).cuda() for v in (pr, ps))
    ctx = A.Context(0)
    scratch = torch.empty(ctx.scratch_bytes(A.MODE_BATCHED, n), dtype=torch.uint8, device="cuda")
    for jo in (0, 1):
        t = ctx.get_tune()
        t.join_order = jo
        ctx.set_tune(t)
        out = torch.full((n,), 0xEE, dtype=torch.uint8, device="cuda")
        ctx.april_filter_pairs_ex(dX, dY, d_r, d_s, n, out, pred, scratch)
        ctx.april_sync_status()
        assert np.array_equal(out.cpu().numpy(), want), jo


@pytest.mark.parametrize("call", ["raw", "packed", "within"])
def test_time_near_windows(torch_cuda, call):
    torch = torch_cuda
    x = np.arange(500, dtype=np.uint64) * 6 + 100
    R, S = (A.april_sets_from_lists(16, [np.stack([x + o, x + o + 1], 1)] * 50, [np.zeros((0, 2))] * 50) for o in (0, 3))
    R.compress(), S.compress()
    dR, dS = A.april_upload(R), A.april_upload(S)
    n = 500_000
    d_r, d_s = (torch.randint(0, 50, (n,), dtype=torch.int32, device="cuda") for _ in range(2))
    ms = []
    for off in (0, 1):
        ctx = _ctx(off)
        out = torch.empty(n, dtype=torch.uint8, device="cuda")
        scratch = torch.empty(ctx.scratch_bytes(A.MODE_BATCHED_PACKED, n), dtype=torch.uint8, device="cuda")
        t = []
        for _ in range(5):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            torch.cuda.synchronize()
            a.record()
            if call == "within":
                ctx.april_filter_pairs_ex(dR, dS, d_r, d_s, n, out, A.PREDICATE_WITHIN, scratch)
            else:
                ctx.april_filter_pairs(dR, dS, d_r, d_s, n, out,
                                       A.MODE_BATCHED if call == "raw" else A.MODE_BATCHED_PACKED, scratch)
            b.record()
            torch.cuda.synchronize()
            t.append(a.elapsed_time(b))
        ctx.april_sync_status()
        assert int(out.max()) == 0
        ms.append(min(t[1:]))
    # the rounds before the hand-over are worth half the merge, and the windows run at part of the occupancy
    # (compressed lists stay in the lanes); lanes alone took 7 times as long
    assert ms[0] < 2.5 * ms[1], ms


@pytest.mark.parametrize("call", ["raw", "within"])
def test_windows_wait_runs_out(torch_cuda, data, call):
    """With the wait limit at 0 the lanes leave every pair to the windows, whose waits then give up at once."""
    torch = torch_cuda
    R, S, _, pr, ps = data
    n = len(pr)
    pred = A.PREDICATE_WITHIN if call == "within" else A.PREDICATE_INTERSECTS
    want, _ = A.april_host_filter_ex(R, S, pr, ps, pred)
    dR, dS = A.april_upload(R), A.april_upload(S)
    d_r, d_s = (torch.from_numpy(v.view(np.int32)).cuda() for v in (pr, ps))
    ctx = A.Context(0)
    scratch = torch.empty(ctx.scratch_bytes(A.MODE_BATCHED, n), dtype=torch.uint8, device="cuda")

    def run():
        out = torch.full((n,), 0xEE, dtype=torch.uint8, device="cuda")
        if call == "within":
            ctx.april_filter_pairs_ex(dR, dS, d_r, d_s, n, out, pred, scratch)
        else:
            ctx.april_filter_pairs(dR, dS, d_r, d_s, n, out, A.MODE_BATCHED, scratch)
        torch.cuda.synchronize()
        return out.cpu().numpy()

    try:
        A.april_debug_set_wait_limit(0)
        got = run()
    finally:
        A.april_debug_set_wait_limit(A.WAIT_LIMIT_DEFAULT)
    with pytest.raises(A.AprilError) as e:
        ctx.april_sync_status()
    assert e.value.status == -5 and (got == 0xFF).any()
    assert np.array_equal(run(), want)
    ctx.april_sync_status()
