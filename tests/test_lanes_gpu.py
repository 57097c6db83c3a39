"""The batched filter's default shape on lists at its edges (GPU only): one
lane per pair reads its lists four intervals at a time and their skip index in
units of 128 intervals (compressed: four blocks of 16), joins of very many
alternations go to eight lanes that split the shorter list, and so do all
pairs of a call of few, with 8, 16 or 32 lanes.  Verdicts must equal host
Algorithm 2 on lists whose lengths and offsets sit around those units, on
lists that interleave to the end, on calls around the sizes where the lanes
per pair change, and with the shape off (the lane groups)."""
import numpy as np
import pytest

from paper_2307_01716_gb300 import april as A

pytestmark = pytest.mark.gpu

ORDER = 16
LENGTHS = [1, 2, 3, 4, 5, 15, 16, 17, 31, 33, 63, 64, 65, 127, 128, 129, 255, 257, 1023, 1025, 4100]


def _lists(rng):
    """Lists of every edge length, spread wide or packed into a band, the last ending at 2^32 now and then; F
    drawn from A's intervals."""
    a, f = [], []
    for n in LENGTHS * 3:
        lo, span = int(rng.integers(0, 1 << 31)), int(rng.choice([8 * n, 64 * n, 1 << 31]))
        p = np.sort(rng.choice(span, 2 * n, replace=False) if span < 1 << 20 else
                    np.unique(rng.integers(0, span, 2 * n + 8))[:2 * n]) + lo
        iv = p.reshape(-1, 2).astype(np.uint64)
        keep = np.ones(len(iv), bool)
        keep[1:] = iv[1:, 0] > iv[:-1, 1]
        iv = iv[keep]
        if rng.random() < 0.2:
            iv[-1, 1] = 1 << 32
        a.append(iv)
        f.append(iv[rng.random(len(iv)) < rng.choice([0.0, 0.1, 0.9])])
    return a, f


def _interleaved(k, hit_at):
    """Two lists of k single cells in turn that share one cell only, at place hit_at (none: -1)."""
    x = np.arange(k, dtype=np.uint64) * 6 + 100
    y = x + 3
    if hit_at >= 0:
        y[hit_at] = x[hit_at]
    return np.stack([x, x + 1], 1), np.stack([y, y + 1], 1)


def _run(torch, R, S, pr, ps, mode, off):
    ctx = A.Context(0)
    t = ctx.get_tune()
    t.triage_off = off
    ctx.set_tune(t)
    n = len(pr)
    d_r, d_s = (torch.from_numpy(v.view(np.int32)).cuda() for v in (pr, ps))
    out = torch.full((n,), 0xEE, dtype=torch.uint8, device="cuda")
    scratch = torch.empty(ctx.scratch_bytes(mode, n), dtype=torch.uint8, device="cuda")
    ctx.april_filter_pairs(R, S, d_r, d_s, n, out, mode, scratch)
    ctx.april_sync_status()
    return out.cpu().numpy()


def _case(packed):
    rng = np.random.default_rng(12)
    (ra, rf), (sa, sf) = _lists(rng), _lists(rng)
    for k, at in ((700, -1), (700, 699), (3000, -1), (3000, 1500), (3000, 2999)):
        x, y = _interleaved(k, at)
        ra.append(x), sa.append(y), rf.append(x[:0]), sf.append(y[::2])
    R, S = A.april_sets_from_lists(ORDER, ra, rf), A.april_sets_from_lists(ORDER, sa, sf)
    g = np.indices((len(ra), len(sa))).reshape(2, -1).astype(np.uint32)
    pr, ps = np.ascontiguousarray(g[0]), np.ascontiguousarray(g[1])
    want, _ = A.april_host_filter(R, S, pr, ps)
    assert (np.bincount(want, minlength=3) > 50).all()
    if packed:
        R.compress()
        S.compress()
    return A.april_upload(R), A.april_upload(S), pr, ps, want


@pytest.mark.parametrize("packed", [False, True])
def test_lane_edges(packed):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dR, dS, pr, ps, want = _case(packed)
    mode = A.MODE_BATCHED_PACKED if packed else A.MODE_BATCHED
    # one call of few pairs, one with a lane per pair, the lane groups
    for off, k in ((0, 1), (0, 17), (1, 1)):
        got, w = _run(torch, dR, dS, np.tile(pr, k), np.tile(ps, k), mode, off), np.tile(want, k)
        bad = np.flatnonzero(got != w)
        assert len(bad) == 0, (off, k, len(bad), [(pr[b % len(pr)], ps[b % len(pr)]) for b in bad[:5]])


def test_call_sizes():
    """Calls around the sizes that change the pairs per warp (w warps of five CTAs per SM: w, 2 w, 4 w) and end
    the few (8 w), by both filters; an id out of range reads as an error and harms no other pair."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dR, dS, pr, ps, want = _case(False)
    w = torch.cuda.get_device_properties(0).multi_processor_count * 5 * 8
    rng = np.random.default_rng(3)
    ctx = A.Context(0)
    for n in (1, 5, 33, w - 1, w, w + 1, 2 * w, 2 * w + 1, 3 * w + 1, 4 * w, 4 * w + 1, 8 * w, 8 * w + 1):
        q = rng.integers(0, len(pr), n)
        d_r, d_s = (torch.from_numpy(v[q].view(np.int32)).cuda() for v in (pr, ps))
        scratch = torch.full((ctx.scratch_bytes(A.MODE_BATCHED, n),), 0xA5, dtype=torch.uint8, device="cuda")
        for broken in (False, True):
            exp = want[q].copy()
            if broken:
                d_r[n // 2] = 0x7FFFFFFF
                exp[n // 2] = A.VERDICT_ERROR
            for ex in (False, True):
                out = torch.full((n,), 0xEE, dtype=torch.uint8, device="cuda")
                if ex:
                    ctx.april_filter_pairs_ex(dR, dS, d_r, d_s, n, out, A.PREDICATE_INTERSECTS, scratch)
                else:
                    ctx.april_filter_pairs(dR, dS, d_r, d_s, n, out, A.MODE_BATCHED, scratch)
                if broken:
                    with pytest.raises(A.AprilError):
                        ctx.april_sync_status()
                else:
                    ctx.april_sync_status()
                assert (out.cpu().numpy() == exp).all(), (n, broken, ex)


@pytest.mark.parametrize("packed", [False, True])
@pytest.mark.parametrize("memory", ["pageable", "pinned", "offset", "unaligned"])
def test_host_pairs(memory, packed):
    """Pairs in host memory of each kind: page-locked ones are read in place (from an odd word of their allocation
    too), others and unaligned ones are copied in; calls of few pairs, of one chunk and of several."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dR, dS, pr, ps, want = _case(packed)
    mode = A.MODE_BATCHED_PACKED if packed else A.MODE_BATCHED
    ctx = A.Context(0)
    rng = np.random.default_rng(4)
    at = {"pageable": 0, "pinned": 0, "offset": 4, "unaligned": 1}[memory]

    def host(v):
        t = torch.empty(4 * len(v) + 8, dtype=torch.uint8)
        t = t if memory == "pageable" else t.pin_memory()
        t = t[at:at + 4 * len(v)]
        t.copy_(torch.from_numpy(v.view(np.uint8)))
        return t

    for n in (1, 3_000, 100_001, 700_001):
        q = rng.integers(0, len(pr), n)
        h_r, h_s = host(pr[q]), host(ps[q])
        out = torch.full((n,), 0xEE, dtype=torch.uint8)
        work = torch.empty(ctx.host_work_bytes(mode, n), dtype=torch.uint8, device="cuda")
        ctx.april_filter_pairs_host(dR, dS, h_r, h_s, n, out, mode, work)
        assert (out.numpy() == want[q]).all(), n
        h_r[4 * (n // 2):4 * (n // 2) + 4] = 0x7F
        with pytest.raises(A.AprilError):
            ctx.april_filter_pairs_host(dR, dS, h_r, h_s, n, out, mode, work)
        assert out.numpy()[n // 2] == A.VERDICT_ERROR
