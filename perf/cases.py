"""Timed workloads of the APRIL filter, one per way a program uses it.

Each case draws two layers of star polygons on the GPU (the distributions of
`synth/configs.py` and `synth/selection.py`: log-normal or Pareto radii, log-
normal vertex counts, 5% of the centres in hotspots), joins their MBRs to the
candidate pairs a spatial join hands to the filter, keeps the layers resident
as a program would (host-built and uploaded, or built on the GPU), and times
one call of a public entry point over them.

A layer of fewer polygons than its full size is a region of the same map: the
centres fill a square in proportion, so that list lengths and pairs per polygon
stay those of the full map.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2307_01716_gb300 import april as A

LATTICE = 1 << 24
DEV = "cuda"

# full size of a layer, candidate pairs per polygon of R that its MBR join
# surely yields (less than the mean: hotspots differ by seed), mean vertices,
# and mean touched cells per polygon of the order-16 grid (rough)
FULL = {"tiny": 1_000, "paper": 200_000, "skewed": 340_000, "county": 1_000}
PAIRS_PER = {"tiny": 1.2, "paper": 10.0, "skewed": 24.0}
VERTS_PER = {"tiny": 110, "paper": 70, "skewed": 50, "county": 540}
CELLS_PER = {"tiny": 16_000, "paper": 1_100, "skewed": 1_300, "county": 76_000}


def listed():
    return [
        # the smallest join: 1,000 x 1,000 polygons on a 2^12 grid; latency and launches
        {"name": "tiny", "kind": "filter", "shape": "tiny", "polys": 1_000, "pairs": 1_187, "order": 12,
         "built": "host", "entry": "batched"},
        # the ordinary join of two map layers: 200k x 200k on a 2^16 grid, sets uploaded from the host
        {"name": "paper", "kind": "filter", "shape": "paper", "polys": 200_000, "pairs": 2_000_000, "order": 16,
         "built": "host", "entry": "batched"},
        # the largest: Pareto radii, lists of 1 to 10^5 intervals, sets built on the GPU
        {"name": "skewed", "kind": "filter", "shape": "skewed", "polys": 340_000, "pairs": 8_000_000, "order": 16,
         "built": "device", "entry": "batched"},
        # space partitioning (Sec. 5.2): each partition on its own 2^14 grid, pairs routed
        {"name": "partitioned", "kind": "partitioned", "shape": "paper", "polys": 60_000, "pairs": 599_999,
         "order": 14, "parts": 16, "packed": False},
        # the same with compressed lists (Sec. 5.1), for sets that have to stay small
        {"name": "packed", "kind": "partitioned", "shape": "paper", "polys": 60_000, "pairs": 599_999,
         "order": 14, "parts": 16, "packed": True},
        # end to end: candidate pairs in pinned host memory in, verdicts in host memory out
        {"name": "host", "kind": "host", "shape": "paper", "polys": 200_000, "pairs": 2_000_000, "order": 16,
         "built": "device"},
        # within join (Sec. 4.3.2) of two layers
        {"name": "within", "kind": "ex", "shape": "paper", "polys": 120_000, "pairs": 1_200_001, "order": 16,
         "order_s": 16, "built": "device", "predicate": "within"},
        # layers rasterised at different granularity (Sec. 5.3)
        {"name": "mixed", "kind": "ex", "shape": "paper", "polys": 120_000, "pairs": 1_200_001, "order": 16,
         "order_s": 14, "built": "device", "predicate": "intersects"},
        # constructing a layer's approximations on the GPU: many small polygons
        {"name": "build-layer", "kind": "build", "shape": "paper", "polys": 200_000, "order": 16},
        # constructing query polygons at query time: few large ones
        {"name": "build-queries", "kind": "build", "shape": "county", "polys": 1_000, "order": 16},
        # selection queries (Sec. 4.3.1): county-like polygons against a resident, indexed layer
        {"name": "select", "kind": "select", "shape": "paper", "polys": 200_000, "queries": 1_000, "order": 16},
        # serving: requests of uneven size against resident layers, several in flight
        {"name": "serve", "kind": "serve", "shape": "skewed", "polys": 300_000, "requests": 24, "lo": 1_000,
         "hi": 1_000_000, "order": 16},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["filter", "filter", "filter", "partitioned", "host", "ex", "ex", "build", "build", "select",
                       "serve"])
    shape = rng.choice(["paper", "skewed"])
    c = {"kind": kind, "shape": shape}
    if kind == "build":
        c["shape"] = rng.choice(["paper", "skewed", "county"])
        hi = {"paper": 190_000, "skewed": 190_000, "county": 900}[c["shape"]]
        c["polys"] = _log_int(rng, {"paper": 2_000, "skewed": 2_000, "county": 7}[c["shape"]], hi)
        c["order"] = rng.randint(12, 16)
        return c
    if kind == "select":
        c.update(shape="paper", polys=_log_int(rng, 5_000, 190_000), queries=_log_int(rng, 20, 1_500),
                 order=rng.randint(14, 16))
        return c
    if kind == "serve":
        c.update(shape="skewed", polys=_log_int(rng, 50_000, 300_000), requests=rng.randint(3, 23),
                 lo=_log_int(rng, 300, 3_000), hi=_log_int(rng, 30_000, 600_000), order=16)
        return c
    if kind == "partitioned":
        c["shape"] = "paper"
        c["polys"] = _log_int(rng, 3_000, 55_000)
        c["parts"] = rng.choice([4, 8, 16])
        c["order"] = rng.randint(12, 14)
        c["packed"] = rng.random() < 0.5
    else:
        c["polys"] = _log_int(rng, 1_000, 250_000)
        c["order"] = rng.choice([13, 14, 15, 16, 16, 16])
        # the host builder takes seconds on a large layer: those come from the GPU builder
        c["built"] = "host" if c["polys"] < 40_000 and rng.random() < 0.6 else "device"
    most = int(c["polys"] * PAIRS_PER[c["shape"]])
    c["pairs"] = _log_int(rng, max(most // 8, 500), most)
    if kind == "filter":
        c["entry"] = rng.choice(["batched", "batched", "noalloc"]) if c["pairs"] <= A.NOALLOC_MAX_PAIRS else "batched"
    if kind == "ex":
        c["predicate"] = rng.choice(["within", "intersects"])
        c["order_s"] = c["order"] if c["predicate"] == "within" else c["order"] - rng.choice([1, 2, 3])
        if c["predicate"] == "intersects" and rng.random() < 0.4:
            c["order"], c["order_s"] = c["order_s"], c["order"]
    return c


# ----------------------------------------------------------------- inputs
def _normal(g, n):
    return torch.randn(n, generator=g, device=DEV, dtype=torch.float64)


def _uniform(g, *n):
    return torch.rand(*n, generator=g, device=DEV, dtype=torch.float64)


def _hotspots(g, shape, n, full_n):
    if shape not in ("paper", "skewed"):
        return None
    return 0.1 + 0.8 * _uniform(g, max(1, round(32 * n / full_n)), 2)


def _layer(g, shape, n, region=1.0, hot=None):
    """n star polygons on the lattice: (xy int32 (V, 2), off int64 (n + 1,), mbr int64 (n, 4)), on the GPU."""
    cen = _uniform(g, n, 2)
    if hot is not None:
        nh = max(1, round(0.05 * n))
        which = torch.randint(0, len(hot), (nh,), generator=g, device=DEV)
        pick = torch.randperm(n, generator=g, device=DEV)[:nh]
        cen[pick] = hot[which] + 2.5e-4 / region * _normal(g, 2 * nh).view(nh, 2)
    cen = (0.5 + (cen - 0.5) * region).clamp(1e-6, 1 - 1e-6)
    if shape == "tiny":
        rad = 0.005 * torch.exp(0.8 * _normal(g, n))
        nv = torch.randint(20, 201, (n,), generator=g, device=DEV)
    elif shape == "county":
        rad = (0.005 * torch.exp(0.6 * _normal(g, n))).clamp(max=0.03)
        nv = (400 * torch.exp(0.8 * _normal(g, n))).round().clamp(32, 5_000).long()
    else:
        if shape == "skewed":
            rad = (2e-4 / 2 ** (1 / 1.3) * (1.0 - _uniform(g, n)) ** (-1 / 1.3)).clamp(max=0.04)
        else:
            rad = (2e-4 * torch.exp(1.2 * _normal(g, n))).clamp(max=0.05)
        nv = (60 * torch.exp(_normal(g, n))).round().clamp(8, 20_000).long()
    # neighbouring vertices stay a few lattice units apart
    nv = torch.minimum(nv, (2 * math.pi * rad * LATTICE / 16).long().clamp(min=8))
    off = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(nv, 0, out=off[1:])
    total = int(off[-1])
    seg = torch.repeat_interleave(torch.arange(n, device=DEV), nv, output_size=total)
    k = torch.arange(total, device=DEV) - off[seg]
    ang = (k + 0.1 + 0.8 * _uniform(g, total)) / nv[seg] + _uniform(g, n)[seg]
    r = rad[seg] * (0.6 + 0.8 * _uniform(g, total))
    d = torch.stack([torch.cos(2 * math.pi * ang) * r, torch.sin(2 * math.pi * ang) * r], 1)
    c = cen[seg]
    # a vertex that would leave the map is pulled towards the centre
    room = torch.where(d > 0, (1.0 - c) / d, torch.where(d < 0, -c / d, torch.full_like(d, math.inf)))
    t = room.amin(1).clamp(max=1.0)
    xy = ((c + t[:, None] * d) * LATTICE).round().clamp(0, LATTICE).to(torch.int32)
    i2 = seg[:, None].expand(-1, 2)
    lo = torch.full((n, 2), LATTICE, dtype=torch.int32, device=DEV).scatter_reduce(0, i2, xy, "amin")
    hi = torch.zeros((n, 2), dtype=torch.int32, device=DEV).scatter_reduce(0, i2, xy, "amax")
    return xy.contiguous(), off, torch.cat([lo, hi], 1).long()


def _copies(mbr, tb):
    """(object, tile) of every tile an MBR meets, by tile, then by object."""
    side = 1 << (25 - tb)
    t0, t1 = mbr[:, :2] >> tb, mbr[:, 2:] >> tb
    w = t1 - t0 + 1
    cnt = w[:, 0] * w[:, 1]
    obj = torch.repeat_interleave(torch.arange(len(mbr), device=DEV), cnt)
    k = torch.arange(len(obj), device=DEV) - (torch.cumsum(cnt, 0) - cnt)[obj]
    tile = (t0[obj, 1] + k // w[obj, 0]) * side + t0[obj, 0] + k % w[obj, 0]
    tile, o = torch.sort(tile, stable=True)
    return obj[o], tile, side


def _candidates(g, mr, ms, most):
    """The MBR join's pairs, tile by tile (each from the tile of its reference
    point), a seeded sample of at most `most` in that order; int32 ids."""
    ext = torch.cat([mr[:, 2:] - mr[:, :2], ms[:, 2:] - ms[:, :2]]).flatten().sort().values
    tb = min(max(int(ext[int(0.9 * (len(ext) - 1))]).bit_length() + 1, 10), 24)
    ro, rt, side = _copies(mr, tb)
    so, st, _ = _copies(ms, tb)
    b = torch.searchsorted(st, rt)
    cnt = torch.searchsorted(st, rt, right=True) - b
    first = torch.cumsum(cnt, 0) - cnt
    copy = torch.repeat_interleave(torch.arange(len(ro), device=DEV), cnt)
    s = so[b[copy] + torch.arange(len(copy), device=DEV) - first[copy]]
    r, tile = ro[copy], rt[copy]
    a, c = mr[r], ms[s]
    low = torch.maximum(a[:, :2], c[:, :2])
    keep = (low <= torch.minimum(a[:, 2:], c[:, 2:])).all(1) & ((low[:, 1] >> tb) * side + (low[:, 0] >> tb) == tile)
    r, s = r[keep], s[keep]
    if len(r) > most:
        pick = torch.randperm(len(r), generator=g, device=DEV)[:most].sort().values
        r, s = r[pick], s[pick]
    return r.to(torch.int32), s.to(torch.int32)


def _cells(case):
    """Touched cells per polygon, roughly: its outline's, and at least one or two per vertex."""
    return CELLS_PER[case["shape"]] * 2.0 ** (case["order"] - 16) + 1.5 * VERTS_PER[case["shape"]]


def _host(layer):
    return layer[0].cpu().numpy(), layer[1].cpu().numpy()


def _resident(ctx, layer, order, built):
    if built == "host":
        return A.april_upload(A.april_build_sets(*_host(layer), A.global_grid(order)))
    return ctx.april_build_sets_device(layer[0], layer[1], A.global_grid(order))[0]


def _bytes(n):
    return torch.empty(max(int(n), 256), dtype=torch.uint8, device=DEV)


def _two_layers(g, case):
    n, shape = case["polys"], case["shape"]
    region = min(1.0, math.sqrt(n / FULL[shape]))
    hot = _hotspots(g, shape, n, FULL[shape])
    return _layer(g, shape, n, region, hot), _layer(g, shape, n, region, hot)


def prepare(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    kind, ctx = case["kind"], A.Context(0)
    st = {"case": case, "ctx": ctx}
    if kind == "build":
        xy, off, _ = _layer(g, case["shape"], case["polys"])
        grid = A.global_grid(case["order"])
        # buffers of a size that the program has found out once; slots that no list uses stay zero
        info = ctx.april_build_sets_device(xy, off, grid)[1]
        room = int(case["polys"] * _cells(case) * (1.6 + 8 / math.sqrt(case["polys"]))) * 17
        st.update(xy=xy, off=off, grid=grid, work=_bytes(info.work_bytes),
                  image=torch.zeros(max(int(info.image_bytes), room), dtype=torch.uint8, device=DEV))
        return st
    if kind == "select":
        data = _layer(g, "paper", case["polys"], 1.0, _hotspots(g, "paper", case["polys"], FULL["paper"]))
        sets = A.april_build_sets(*_host(data), A.global_grid(case["order"]))
        q = _layer(g, "county", case["queries"])
        st.update(R=A.april_upload(sets), index=A.april_index_upload(A.april_index_build(sets)),
                  Q=_resident(ctx, q, case["order"], "device"))
        cap = 1 << max(14, int(case["polys"] * case["queries"] * 1e-3).bit_length())
        st.update(cap=cap, r=torch.zeros(cap, dtype=torch.int32, device=DEV),
                  q=torch.zeros(cap, dtype=torch.int32, device=DEV), v=torch.zeros(cap, dtype=torch.uint8, device=DEV),
                  qoff=torch.empty(case["queries"] + 1, dtype=torch.int32, device=DEV),
                  scratch=_bytes(ctx.select_scratch_bytes(cap)))
        return st
    lr, ls = _two_layers(g, case)
    most = case["pairs"] if "pairs" in case else int(case["polys"] * PAIRS_PER[case["shape"]])
    r, s = _candidates(g, lr[2], ls[2], most)
    n = len(r)
    if kind == "partitioned":
        hr, hs = A.april_build_partitioned_sets(*_host(lr), *_host(ls), case["parts"], case["order"])
        if case["packed"]:
            hr.compress()
            hs.compress()
        st.update(R=A.april_upload(hr), S=A.april_upload(hs),
                  mode=A.MODE_BATCHED_PACKED if case["packed"] else A.MODE_BATCHED)
    elif kind == "serve":
        st.update(R=_resident(ctx, lr, case["order"], "device"), S=_resident(ctx, ls, case["order"], "device"))
        # sizes spread over the logarithm of their range, in a mixed order; a
        # request's pairs are neighbours in the join's order: a window of the map
        rng = np.random.default_rng(int(seed))
        sizes = np.exp(np.linspace(math.log(case["lo"]), math.log(case["hi"]), case["requests"])).astype(np.int64)
        reqs = []
        for size in np.minimum(np.random.default_rng(case["requests"]).permutation(sizes), n).tolist():
            at = int(rng.integers(0, n - size + 1))
            reqs.append((r[at:at + size].cpu().pin_memory(), s[at:at + size].cpu().pin_memory(),
                         torch.empty(size, dtype=torch.uint8).pin_memory()))
        st.update(reqs=reqs, server=A.Server(ctx, st["R"], st["S"], _bytes(1 << 30), 8))
        return st
    else:
        st.update(R=_resident(ctx, lr, case["order"], case["built"]),
                  S=_resident(ctx, ls, case.get("order_s", case["order"]), case["built"]), mode=A.MODE_BATCHED)
    if kind == "host":
        st.update(n=n, r=r.cpu().pin_memory(), s=s.cpu().pin_memory(), out=torch.empty(n, dtype=torch.uint8).pin_memory(),
                  work=_bytes(ctx.host_work_bytes(A.MODE_BATCHED, n)))
        return st
    st.update(n=n, r=r, s=s, out=torch.empty(n, dtype=torch.uint8, device=DEV),
              scratch=_bytes(ctx.scratch_bytes(st["mode"], n)))
    return st


# ------------------------------------------------------------------- pass
def run(st):
    case, ctx = st["case"], st["ctx"]
    kind = case["kind"]
    if kind == "build":
        ctx.april_build_sets_device(st["xy"], st["off"], st["grid"], st["work"], st["image"])
        return st["image"]
    if kind == "select":
        m = ctx.april_select(st["index"], st["R"], st["Q"], st["cap"], st["r"], st["q"], st["v"], st["qoff"],
                             st["scratch"])
        return {"pairs": m, "r": st["r"], "q": st["q"], "verdict": st["v"], "off": st["qoff"]}
    if kind == "serve":
        tickets = [st["server"].april_submit(*req) for req in st["reqs"]]
        for t in tickets:
            st["server"].april_wait(t)
        return [req[2] for req in st["reqs"]]
    if kind == "host":
        ctx.april_filter_pairs_host(st["R"], st["S"], st["r"], st["s"], st["n"], st["out"], A.MODE_BATCHED, st["work"])
    elif kind == "ex":
        pred = A.PREDICATE_WITHIN if case["predicate"] == "within" else A.PREDICATE_INTERSECTS
        ctx.april_filter_pairs_ex(st["R"], st["S"], st["r"], st["s"], st["n"], st["out"], pred, st["scratch"])
    elif kind == "filter" and case["entry"] == "noalloc":
        A.april_filter_pairs_noalloc(st["R"], st["S"], st["r"], st["s"], st["n"], st["out"])
    else:
        ctx.april_filter_pairs(st["R"], st["S"], st["r"], st["s"], st["n"], st["out"], st["mode"], st["scratch"])
    return st["out"]


def work(case):
    """Bytes one pass cannot do without.  Filter: per pair its two ids and its
    verdict, and one 32-byte sector of each of its two objects' descriptors
    and of the two lists a verdict rests on.  Build: the vertices read, the
    descriptors, MBRs and (about half a list interval per touched cell and
    list) the intervals written.  The work is integer compare and merge: no
    floating-point operations."""
    kind = case["kind"]
    if kind == "build":
        return {"bytes": case["polys"] * (8 * VERTS_PER[case["shape"]] + 32 + 0.5 * _cells(case) * 2 * 8), "flops": 0}
    if kind == "select":
        pairs = case["polys"] * case["queries"] * 4.2e-4
        return {"bytes": pairs * (8 + 1 + 4 * 32) + case["queries"] * 20 + case["polys"] * 20, "flops": 0}
    if kind == "serve":
        mean = (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        return {"bytes": case["requests"] * mean * (8 + 1 + 4 * 32), "flops": 0}
    return {"bytes": case["pairs"] * (8 + 1 + 4 * 32), "flops": 0}


def exact(case, seed):
    return None  # every output is a whole number
