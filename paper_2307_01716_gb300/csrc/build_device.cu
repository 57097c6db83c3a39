// GPU construction of APRIL approximations: polygons in device memory in,
// a device image of their A- and F-lists (the layout the filter reads) out.
//
// The cells and lists are exactly the host builder's (build_sets.cpp): both
// take their arithmetic from geom.h (raster.h restates the edge arithmetic in
// 32 bits), and the lists are canonical (maximal intervals of the A and F cell
// sets, Sec. 4.1), so the two agree list for list.  The steps:
//   count (k_bcount, k_bcount_big): MBR, the number of touched-cell incidences
//          T (cells an edge meets, per edge) and of centre-line incidences;
//   place (k_bsum, k_btop, k_bplace): every polygon's slot range (in polygon
//          order) and the path it takes; the host reads the totals once;
//   raster (k_bsmall, k_bmid, k_btile): a window of cells as bitmaps in
//          shared memory.  Every edge sets, row by row, the bits of the cells
//          it touches and of those it enters, and flips the bit from which on
//          the row's cell centres lie on its other side; a prefix XOR along
//          the rows then tells the cells whose centre is inside.  F is inside
//          and not entered, A is touched or F.  The bitmaps are read back in
//          Hilbert order, an 8 x 8 block at a time, and the places where a
//          bit differs from the one before start and end the intervals.
// A window of up to 64 x 64 cells is a warp's (k_bsmall), up to 256 x 256 a
// CTA's (k_bmid); larger polygons are cut into the Hilbert-aligned tiles of
// 256 x 256 cells of their window, each of which walks all of the polygon's
// edges and finds the intervals started before it by looking back over the
// records of the tiles before it.  No cell is sorted: the work is per cell row
// an edge meets, per block of the window and, with tiles, per tile and edge.
//   A polygon whose outline meets few cells for the tiles of its window and
// its vertices (or whose coordinates do not fit raster.h) is built from its
// sorted cells instead, where empty tiles and edges elsewhere cost nothing
// (path_of has the line):
//   emit   (k_bemit, one CTA per polygon, persistent): every edge writes its
//          touched cells as keys (polygon << 33 | Hilbert id << 1 | crossed),
//          the crossed flag saying whether the edge enters the cell's open
//          square;
//   sort   (k_rs_*): one stable LSD radix sort of all keys of all such
//          polygons (8-bit digits, the passes the key width needs), so that
//          every polygon's keys end up sorted in its own range;
//   build  (k_bconstruct, one CTA per polygon, persistent):
//     2. the sorted keys are reduced to one key per cell (crossed if any
//        edge crossed it);
//     3. the sorted crossings of every cell row's centre line (k_bemit writes
//        one key per edge and row it crosses: polygon, row, floor of the
//        crossing's x; the same radix sort orders them) give each row's
//        crossing list;
//     4. one point-in-polygon test at the first cell of every gap between
//        consecutive touched ids (a gap is wholly inside or outside: Sec.
//        6.2) and at every touched cell no edge crosses (Full when its
//        centre is inside): the parity of the row's crossings right of the
//        centre, by binary search;
//     5. the A- and F-intervals come out of block scans over the cells:
//        an A interval breaks at a non-empty gap outside the polygon, an F
//        interval runs over consecutive Full gaps and cells.
// Each polygon's lists go to a slot range sized from T (|A| <= T and
// |F| <= T + 1), so no second pass is needed; unused slots stay unused.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <string>

#include "april_internal.h"
#include "geom.h"
#include "raster.h"

using april::fail;
using namespace april_geom;

namespace {

constexpr uint32_t kFull = 0xffffffffu;
constexpr unsigned kBB = 256;  // build CTA size
constexpr unsigned kBW = kBB / 32;
constexpr uint32_t kStatusTimeout = 2u;  // the context status word's bit for a bounded wait that ran out

struct GridP {
    int64_t ox, oy, h, G;
    uint32_t order;
};

// Per polygon, written by the count and place steps.
struct PolyMeta {
    uint64_t slot_off;   // into the image's interval slots
    uint64_t key_off;    // sorted path: into the key and temp arrays (keys)
    uint64_t rb_off;     // sorted path: into the row-start array (uint32, rows + 1)
    uint64_t cross_off;  // sorted path: into the crossing-key arrays (keys)
    uint32_t T;          // touched-cell incidences
    uint32_t inc;        // centre-line incidences
    int32_t mbr[4];
    uint32_t err;        // 0 ok; 1 fewer than 3 vertices; 2 outside the grid; 3 too large; 4 meets no cell;
                         // kTileFailed (set by k_btile)
    uint32_t item_off;   // tiled path: its first tile record
};
static_assert(sizeof(PolyMeta) == 64, "the work layout counts 80 bytes per polygon: the record and four list entries");

// The path a polygon takes.
enum : uint32_t { kSmall = 0, kMid = 1, kTiled = 2, kSorted = 3, kPaths = 4 };

struct Totals {
    unsigned long long keys, rb, slots, cross;  // over all polygons
    unsigned long long first_err;               // polygon << 8 | err of the first rejected one
    unsigned long long tiled;                   // polygons << 40 | tile records
    unsigned long long skeys, srb, scross;      // of the sorted path
    unsigned long long big;                     // polygons << 40 | chunks of their edges
    unsigned long long gain;                    // what sorting saves over tiles (tiles_cost_more), in all
    unsigned int n_err, count[kPaths];
    unsigned int ctr_emit, ctr_build, ctr_count, ctr_tile;  // persistent kernels' polygon counters
};
static_assert(sizeof(Totals) <= 256, "the work layout keeps 256 bytes for the totals");

// Crossing keys: polygon << 42 | (row - wj0) << 26 | (floor(x) - xmn), the x
// of an edge's crossing with the row's centre line (26 bits cover the
// lattice square and its margins).
constexpr uint32_t kCrossXBits = 26, kCrossRowBits = 16, kCrossPolyShift = kCrossXBits + kCrossRowBits;

// The window of cells a polygon's MBR meets.
struct CellWin {
    int64_t wi0, wj0, wi1, wj1;
};
__device__ __forceinline__ CellWin window_of(const int32_t *mbr, const GridP &g) {
    CellWin w;
    cell_window(mbr[0], mbr[1], mbr[2], mbr[3], g.ox, g.oy, g.h, g.G, w.wi0, w.wj0, w.wi1, w.wj1);
    return w;
}

__device__ __forceinline__ uint64_t even_up(uint64_t v) { return (v + 1) & ~1ull; }

__device__ __forceinline__ int2 vtx(const int2 *xy, uint64_t b, uint64_t nv, uint64_t k) {
    return xy[b + (k == nv ? 0 : k)];
}

// -------------------------------------------------- teams of 32 or 256 threads
// A warp, or a CTA of 256 threads, working on one polygon (or one tile).
template <uint32_t NT>
struct Team {
    static __device__ __forceinline__ uint32_t rank() { return NT == 32 ? (threadIdx.x & 31u) : threadIdx.x; }
    static __device__ __forceinline__ void sync() {
        if (NT == 32) __syncwarp();
        else __syncthreads();
    }
    // Exclusive sum over the team; `sums` holds NT / 32 words.
    static __device__ __forceinline__ uint32_t scan(uint32_t v, uint32_t &total, uint32_t *sums) {
        const uint32_t lane = threadIdx.x & 31u;
        uint32_t x = v;
#pragma unroll
        for (uint32_t d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(kFull, x, d);
            if (lane >= d) x += y;
        }
        if (NT == 32) {
            total = __shfl_sync(kFull, x, 31);
            return x - v;
        }
        if (lane == 31) sums[threadIdx.x >> 5] = x;
        __syncthreads();
        uint32_t before = 0, all = 0;
#pragma unroll
        for (uint32_t w = 0; w < NT / 32; ++w) {
            if (w < (threadIdx.x >> 5)) before += sums[w];
            all += sums[w];
        }
        __syncthreads();
        total = all;
        return before + x - v;
    }
};

// The rows an edge meets come in items of up to kRowRun, so that a team's
// threads share them evenly whatever the edges' lengths: NT edges at a time
// wait in shared memory with the items before each.  An item costs two
// divisions, and long ones leave threads waiting for each other: 1,000 query
// polygons of long edges took 3.04 ms with runs of 4, 2.88 with 8 or 16 and
// 3.31 with 32; 200,000 layer polygons 9.69, 9.55, 9.95 and 10.9 ms.
constexpr int32_t kRowRun = 8;
template <uint32_t NT>
struct WalkShared {
    EdgeRel ed[NT];
    uint32_t pre[NT];
    uint32_t sums[NT / 32];
};

// Calls row(RowCells) for every (edge, row) of edges [from, to) of the polygon
// with rows in [rlo, rhi], for the edges pre(edge) takes.  Every thread of the team calls it.
template <uint32_t NT, class Pre, class Row>
__device__ __forceinline__ void walk_edges(const int2 *__restrict__ xy, uint64_t b, uint64_t nv, uint64_t from,
                                           uint64_t to, const GridP &g, int l, int32_t rlo, int32_t rhi,
                                           WalkShared<NT> &ws, Pre pre, Row row) {
    const uint32_t t = Team<NT>::rank();
    const int32_t ox = (int32_t)g.ox, oy = (int32_t)g.oy;
    for (uint64_t e0 = from; e0 < to; e0 += NT) {
        uint32_t cnt = 0;
        if (e0 + t < to) {
            const int2 a = xy[b + e0 + t], c = vtx(xy, b, nv, e0 + t + 1);
            const EdgeRel e = edge_rel(a.x - ox, a.y - oy, c.x - ox, c.y - oy);
            int32_t j0, j1;
            rel_rows(e, l, (int32_t)g.G, j0, j1);
            j0 = max(j0, rlo);
            j1 = min(j1, rhi);
            if (pre(e) && j1 >= j0) cnt = (uint32_t)((j1 - j0) / kRowRun) + 1u;
            ws.ed[t] = e;
        }
        uint32_t total;
        ws.pre[t] = Team<NT>::scan(cnt, total, ws.sums);
        Team<NT>::sync();
        for (uint32_t q = t; q < total; q += NT) {
            uint32_t lo = 0, hi = NT - 1;  // the last edge with at most q items before it
#pragma unroll
            for (uint32_t s = 1; s < NT; s <<= 1) {
                const uint32_t mid = (lo + hi + 1) >> 1;
                if (ws.pre[mid] <= q) lo = mid;
                else hi = mid - 1;
            }
            const EdgeRel e = ws.ed[lo];
            int32_t j0, j1;
            rel_rows(e, l, (int32_t)g.G, j0, j1);
            j0 = max(j0, rlo) + (int32_t)(q - ws.pre[lo]) * kRowRun;
            j1 = min(min(j1, rhi), j0 + kRowRun - 1);
            edge_walk(e, l, j0, j1, row);
        }
        Team<NT>::sync();
    }
}

// ------------------------------------------------------------------ count
// Whether a polygon's coordinates fit raster.h.
__device__ __forceinline__ bool fits_raster(const int32_t *mbr, const GridP &g) {
    constexpr int64_t lim = 1ll << 28;
    return mbr[0] - g.ox > -lim && mbr[1] - g.oy > -lim && mbr[2] - g.ox < lim && mbr[3] - g.oy < lim &&
           g.h <= (1ll << 24);
}

__device__ __forceinline__ void reject(Totals *tot, uint32_t p, uint32_t err) {
    atomicAdd(&tot->n_err, 1u);
    atomicMin(&tot->first_err, (unsigned long long)p << 8 | err);
}

template <uint32_t NT, class T, class Op>
__device__ __forceinline__ T team_reduce(T v, Op op, T *red) {
    for (int o = 16; o; o >>= 1) v = op(v, __shfl_xor_sync(kFull, v, o));
    if (NT == 32) return v;
    if ((threadIdx.x & 31u) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    v = red[0];
    for (uint32_t w = 1; w < NT / 32; ++w) v = op(v, red[w]);
    __syncthreads();
    return v;
}

// The touched-cell and centre-line incidences of edges [from, to) of a
// polygon with window W, summed over the team.
template <uint32_t NT>
__device__ __forceinline__ void count_edges(const int2 *__restrict__ xy, uint64_t b, uint64_t nv, uint64_t from,
                                            uint64_t to, const int32_t *mbr, const GridP &g, int l, WalkShared<NT> &ws,
                                            unsigned long long *red, unsigned long long &T, unsigned long long &inc) {
    const CellWin W = window_of(mbr, g);
    T = inc = 0;
    if (fits_raster(mbr, g)) {
        const int32_t w0 = (int32_t)W.wj0, w1 = (int32_t)W.wj1, gx = (int32_t)g.G - 1;
        uint32_t t32 = 0;  // a thread's share of one batch of rows stays far below 2^32
        walk_edges<NT>(
            xy, b, nv, from, to, g, l, 0, gx, ws,
            [&](const EdgeRel &e) {
                int32_t r0, r1;
                rel_centre_rows(e, l, r0, r1);
                r0 = max(r0, w0), r1 = min(r1, w1);
                if (r1 >= r0) inc += (unsigned long long)(r1 - r0 + 1);
                T += t32;
                t32 = 0;
                return true;
            },
            [&](const RowCells &c) {
                const int32_t i0 = max(c.i0, 0), i1 = min(c.i1, gx);
                if (i1 >= i0) t32 += (uint32_t)(i1 - i0 + 1);
            });
        T += t32;
    } else {
        for (uint64_t k = from + Team<NT>::rank(); k < to; k += NT) {
            const int2 a = vtx(xy, b, nv, k), c = vtx(xy, b, nv, k + 1);
            const EdgeUp e = edge_up(a.x, a.y, c.x, c.y);
            int64_t r0, r1, i0, i1;
            centre_rows(e, g.oy, g.h, W.wj0, W.wj1, r0, r1);
            if (r1 >= r0) inc += (unsigned long long)(r1 - r0 + 1);
            edge_rows(e, g.oy, g.h, g.G, r0, r1);
            for (int64_t j = r0; j <= r1; ++j)
                if (edge_cells_in_row(e, g.ox, g.oy, g.h, g.G, j, i0, i1)) T += (unsigned long long)(i1 - i0 + 1);
        }
    }
    auto sum = [](unsigned long long x, unsigned long long y) { return x + y; };
    T = team_reduce<NT>(T, sum, red);
    inc = team_reduce<NT>(inc, sum, red);
}

// The blocks of 8 x 8 cells (or, with lv = 8, the tiles of 2^8 x 2^8) a window
// covers, and the Hilbert-aligned squares of 2^m x 2^m of them that cover it:
// at most 5 x 5, a quarter of the longer side each, so that at most about half
// of their blocks lie outside (with 2 x 2 squares it was three quarters: the
// window kernels took a third longer).
struct Cover {
    int32_t x0, y0, x1, y1;  // first and last block (tile) columns and rows
    uint32_t m;              // squares of 4^m blocks
    uint32_t nx, n;          // squares in a row, in all
};
__device__ __forceinline__ Cover cover_of(const CellWin &W, int lv) {
    Cover c;
    c.x0 = (int32_t)(W.wi0 >> lv), c.y0 = (int32_t)(W.wj0 >> lv);
    c.x1 = (int32_t)(W.wi1 >> lv), c.y1 = (int32_t)(W.wj1 >> lv);
    const uint32_t side = (uint32_t)max(c.x1 - c.x0, c.y1 - c.y0);  // one less than the longer side
    c.m = side > 3 ? 30u - (uint32_t)__clz(side) : 0u;
    c.nx = (uint32_t)((c.x1 >> c.m) - (c.x0 >> c.m)) + 1u;
    c.n = c.nx * ((uint32_t)((c.y1 >> c.m) - (c.y0 >> c.m)) + 1u);
    return c;
}

// What tiles cost a polygon of nv vertices more than sorting its cells, in
// picoseconds of the whole chip's time (0: they cost less).  Measured over
// smooth and jagged outlines of 50 to 10^6 vertices, windows of 300 to 30,000
// cells and 1 to 20,000 polygons: a tile takes 37 ns and every edge it walks
// past 7 ps, a sorted cell 0.22 ns.  So 100 outlines of 100,000 vertices over
// 535,000 tiles take 354 ms in tiles and 7.7 sorted, but 1,000 query polygons
// of 540 jagged vertices (34,000 tiles, 71M cells) 2.9 and 37.
__device__ __forceinline__ uint64_t tiles_cost_more(const CellWin &W, uint32_t T, uint64_t nv) {
    const Cover tc = cover_of(W, 8);
    const uint64_t tiles = (uint64_t)(tc.x1 - tc.x0 + 1) * (uint64_t)(tc.y1 - tc.y0 + 1);
    const uint64_t tiled = tiles * (37000 + 7 * nv), sorted = 220ull * T;
    return tiled > sorted ? min((unsigned long long)(tiled - sorted), 1ull << 40) : 0;  // sums over 2^22 polygons fit
}

// Where the paths part: a window of at most 8 x 8 blocks is a warp's (three
// bitmaps of 64 x 64 cells are 1.6 KB), at most 32 x 32 a CTA's (28 KB).  A
// larger one is tiled while it has no more tile records (16 bytes each) than
// a quarter of its touched cells, so that the records fit in the work buffer,
// and unless sorting saves time: `gain`, what it saves over all polygons for
// which tiles cost more, has to pay for the sort's launches (1.3 ms) and for
// the one CTA that takes a polygon's cells at 30 ns each while others end
// (1.7M cells of one polygon: 57 ms, 0.7 in tiles).
__device__ __forceinline__ uint32_t path_of(const PolyMeta &m, const GridP &g, uint64_t nv, uint64_t gain,
                                            uint32_t &records) {
    records = 0;
    if (m.T == 0) return kSmall;
    if (!fits_raster(m.mbr, g)) return kSorted;
    const CellWin W = window_of(m.mbr, g);
    const Cover c = cover_of(W, 3);
    const int32_t side = max(c.x1 - c.x0, c.y1 - c.y0) + 1;
    if (side <= 8) return kSmall;
    if (side <= 32) return kMid;
    const Cover tc = cover_of(W, 8);
    records = tc.n << (2 * tc.m);
    if (records > m.T / 4) return kSorted;
    return gain > 1300000000ull + 30000ull * m.T && tiles_cost_more(W, m.T, nv) ? kSorted : kTiled;
}

// A polygon's record once its incidences are known (by one warp).
__device__ __forceinline__ void finish_count(const int2 *__restrict__ xy, uint64_t b, uint64_t nv, uint32_t p,
                                             const GridP &g, PolyMeta &m, unsigned long long T, unsigned long long inc,
                                             PolyMeta *meta, Totals *tot) {
    const uint32_t lane = threadIdx.x & 31u;
    if (T > 0x7FFFFFFFull || inc > 0x7FFFFFFFull) m.err = 3;
    if (!m.err && T == 0) {
        // no edge meets a cell: the polygon holds the whole grid or misses it,
        // which the centre of cell (0, 0) tells (crossing parity)
        const int64_t xc = g.ox + g.h / 2, yc = g.oy + g.h / 2;
        uint32_t par = 0;
        for (uint64_t k = lane; k < nv; k += 32) {
            const int2 a = vtx(xy, b, nv, k), c = vtx(xy, b, nv, k + 1);
            const EdgeUp ed = edge_up(a.x, a.y, c.x, c.y);
            if (ed.ay <= yc && yc < ed.by && turn(ed.ax, ed.ay, ed.bx, ed.by, xc, yc) > 0) par ^= 1u;
        }
        if (!(__popc(__ballot_sync(kFull, par & 1u)) & 1)) m.err = 4;
    }
    if (lane == 0) {
        m.T = m.err ? 0u : (uint32_t)T;
        m.inc = m.err ? 0u : (uint32_t)inc;
        meta[p] = m;
        uint32_t records;
        if (path_of(m, g, nv, 0, records) == kTiled) {
            const uint64_t more = tiles_cost_more(window_of(m.mbr, g), m.T, nv);
            if (more) atomicAdd(&tot->gain, more);
        }
        if (m.err) reject(tot, p, m.err);
    }
    __syncwarp();
}

// A warp per polygon: MBR, incidences, errors.  Polygons of more than
// `big_verts` vertices only get their MBR here and are listed, with the chunks
// of 256 edges that k_bcount_big counts by a CTA each, and k_bcount_end ends
// them.  The walk is integer arithmetic on the edges (8 bytes a vertex read),
// bound by issue: 1.4 ms of the 9.6 that 200,000 layer polygons (14M vertices)
// take in all (one CTA per polygon over expanded edge rows, after a warp's
// count: 3.3 ms).
constexpr uint32_t kChunkEdges = 256;
__global__ void __launch_bounds__(256) k_bcount(const int2 *__restrict__ xy, const uint64_t *__restrict__ off,
                                                uint32_t n, GridP g, int l, PolyMeta *meta, Totals *tot,
                                                uint32_t *big, uint64_t big_verts) {
    __shared__ WalkShared<32> ws[kBW];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    uint32_t p = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;  // the first by place, then by the counter
    const uint32_t warps = gridDim.x * kBW;
    while (p < n) {
        const uint64_t b = off[p], e = off[p + 1], nv = e >= b ? e - b : 0;
        PolyMeta m{};
        if (nv < 3) {
            m.err = 1;
        } else {
            int32_t xmn = INT32_MAX, ymn = INT32_MAX, xmx = INT32_MIN, ymx = INT32_MIN;
            for (uint64_t k = lane; k < nv; k += 32) {
                const int2 v = xy[b + k];
                xmn = min(xmn, v.x), xmx = max(xmx, v.x), ymn = min(ymn, v.y), ymx = max(ymx, v.y);
            }
            for (int o = 16; o; o >>= 1) {
                xmn = min(xmn, __shfl_xor_sync(kFull, xmn, o)), ymn = min(ymn, __shfl_xor_sync(kFull, ymn, o));
                xmx = max(xmx, __shfl_xor_sync(kFull, xmx, o)), ymx = max(ymx, __shfl_xor_sync(kFull, ymx, o));
            }
            m.mbr[0] = xmn, m.mbr[1] = ymn, m.mbr[2] = xmx, m.mbr[3] = ymx;
            const CellWin W = window_of(m.mbr, g);
            if (W.wi0 > W.wi1 || W.wj0 > W.wj1) m.err = 2;
            else if ((int64_t)xmx - xmn >= (1ll << kCrossXBits)) m.err = 3;
        }
        if (m.err) {
            if (lane == 0) {
                meta[p] = m;
                reject(tot, p, m.err);
            }
        } else if (nv > big_verts) {
            if (lane == 0) {  // list place and first chunk by one add, so that both rise together
                const unsigned long long chunks = (nv + kChunkEdges - 1) / kChunkEdges;
                const unsigned long long a = atomicAdd(&tot->big, 1ull << 40 | chunks);
                big[(uint32_t)(a >> 40)] = p;
                m.slot_off = a & ((1ull << 40) - 1);  // until the place step: the first chunk, and T and
                meta[p] = m;                          // inc summed up in key_off and rb_off
            }
        } else {
            unsigned long long T, inc;
            count_edges<32>(xy, b, nv, 0, nv, m.mbr, g, l, ws[warp], nullptr, T, inc);
            finish_count(xy, b, nv, p, g, m, T, inc, meta, tot);
        }
        uint32_t c = 0;
        if (lane == 0) c = atomicAdd(&tot->ctr_count, 1u);
        c = __shfl_sync(kFull, c, 0);
        p = c < n ? min(n, warps + c) : n;
    }
}

__global__ void __launch_bounds__(256) k_bcount_big(const int2 *__restrict__ xy, const uint64_t *__restrict__ off,
                                                    GridP g, int l, PolyMeta *meta, Totals *tot,
                                                    const uint32_t *__restrict__ big) {
    __shared__ WalkShared<256> ws;
    __shared__ unsigned long long red[kBW];
    const unsigned long long all = *((volatile unsigned long long *)&tot->big), chunks = all & ((1ull << 40) - 1);
    const uint32_t n = (uint32_t)(all >> 40);
    for (uint64_t q = blockIdx.x; q < chunks; q += gridDim.x) {
        uint32_t lo = 0, hi = n - 1;  // the last polygon whose first chunk is at most q
        while (lo < hi) {
            const uint32_t mid = (lo + hi + 1) >> 1;
            if (meta[big[mid]].slot_off <= q) lo = mid;
            else hi = mid - 1;
        }
        const uint32_t p = big[lo];
        const uint64_t b = off[p], nv = off[p + 1] - b, from = (q - meta[p].slot_off) * kChunkEdges;
        const int32_t mbr[4] = {meta[p].mbr[0], meta[p].mbr[1], meta[p].mbr[2], meta[p].mbr[3]};
        unsigned long long T, inc;
        count_edges<256>(xy, b, nv, from, min(nv, from + kChunkEdges), mbr, g, l, ws, red, T, inc);
        if (threadIdx.x == 0) {
            atomicAdd((unsigned long long *)&meta[p].key_off, T);
            atomicAdd((unsigned long long *)&meta[p].rb_off, inc);
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(256) k_bcount_end(const int2 *__restrict__ xy, const uint64_t *__restrict__ off,
                                                    GridP g, PolyMeta *meta, Totals *tot,
                                                    const uint32_t *__restrict__ big) {
    const uint32_t n = (uint32_t)(*((volatile unsigned long long *)&tot->big) >> 40);
    for (uint32_t q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < n; q += gridDim.x * kBW) {
        const uint32_t p = big[q];
        PolyMeta m = meta[p];
        __syncwarp();
        finish_count(xy, off[p], off[p + 1] - off[p], p, g, m, m.key_off, m.rb_off, meta, tot);
    }
}

// ------------------------------------------------------------------ place
// Exclusive offsets in polygon order: the slots (a polygon takes 2 even(T + 1):
// |A| <= max(T, 1) and |F| <= T + 1) and, for the sorted path, the keys and the
// crossing keys; the totals, and each polygon's path.  The sort leaves the keys
// in polygon order, so a polygon's range has to lie there too, whatever order
// the blocks run in.  Blocks of kPlace polygons: k_bsum leaves a block's sums
// in its first record, k_btop turns those into offsets, k_bplace does the rest.
constexpr uint32_t kPlace = 2048, kPlacePer = kPlace / 256;
__device__ __forceinline__ uint64_t poly_slots(const PolyMeta &m) { return 2 * even_up((uint64_t)m.T + 1); }

__global__ void __launch_bounds__(256) k_bsum(const uint64_t *__restrict__ off, PolyMeta *meta, uint32_t n, GridP g,
                                              Totals *tot) {
    __shared__ unsigned long long red[kBW];
    const uint64_t gain = tot->gain;
    unsigned long long s[6] = {0, 0, 0, 0, 0, 0};
    for (uint32_t k = 0; k < kPlacePer; ++k) {
        const uint32_t p = blockIdx.x * kPlace + k * 256 + threadIdx.x;
        if (p >= n) break;
        const PolyMeta m = meta[p];
        const CellWin W = window_of(m.mbr, g);
        uint32_t records;
        const bool sorted = !m.err && path_of(m, g, off[p + 1] - off[p], gain, records) == kSorted;
        s[0] += m.T;
        s[1] += m.err ? 0 : (unsigned long long)(W.wj1 - W.wj0 + 2);
        s[2] += poly_slots(m);
        s[3] += m.inc;
        s[4] += sorted ? m.T : 0;
        s[5] += sorted ? m.inc : 0;
    }
    auto sum = [](unsigned long long x, unsigned long long y) { return x + y; };
    for (int f = 0; f < 6; ++f) s[f] = team_reduce<256>(s[f], sum, red);
    if (threadIdx.x == 0) {
        atomicAdd(&tot->keys, s[0]);
        atomicAdd(&tot->rb, s[1]);
        atomicAdd(&tot->cross, s[3]);
        PolyMeta &first = meta[blockIdx.x * kPlace];
        first.slot_off = s[2], first.key_off = s[4], first.cross_off = s[5];
    }
}

__global__ void __launch_bounds__(1024) k_btop(PolyMeta *meta, uint32_t nblocks, Totals *tot) {
    __shared__ unsigned long long s_w[32];
    const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5;
    auto offsets = [&](uint64_t PolyMeta::*field) {
        unsigned long long base = 0;
        for (uint32_t b0 = 0; b0 < nblocks; b0 += 1024) {
            const bool on = b0 + t < nblocks;
            const unsigned long long v = on ? meta[(uint64_t)(b0 + t) * kPlace].*field : 0ull;
            unsigned long long x = v;
            for (uint32_t d = 1; d < 32; d <<= 1) {
                const unsigned long long y = __shfl_up_sync(kFull, x, d);
                if (lane >= d) x += y;
            }
            if (lane == 31) s_w[warp] = x;
            __syncthreads();
            unsigned long long before = base, all = base;
            for (uint32_t w = 0; w < 32; ++w) {
                if (w < warp) before += s_w[w];
                all += s_w[w];
            }
            __syncthreads();
            if (on) meta[(uint64_t)(b0 + t) * kPlace].*field = before + x - v;
            base = all;
        }
        return base;
    };
    const unsigned long long slots = offsets(&PolyMeta::slot_off), keys = offsets(&PolyMeta::key_off),
                             cross = offsets(&PolyMeta::cross_off);
    if (t == 0) tot->slots = slots, tot->skeys = keys, tot->scross = cross;
}

__global__ void __launch_bounds__(256) k_bplace(const uint64_t *__restrict__ off, PolyMeta *meta, uint32_t n, GridP g,
                                                Totals *tot, uint32_t *lists) {
    __shared__ unsigned long long s_w[kBW];
    const uint64_t gain = tot->gain;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const PolyMeta &block = meta[blockIdx.x * kPlace];
    unsigned long long base = block.slot_off, kbase = block.key_off, cbase = block.cross_off;
    __syncthreads();
    // exclusive sum over the block from `from` on, which becomes the next start
    auto scan = [&](unsigned long long v, unsigned long long &from) {
        unsigned long long x = v;
        for (uint32_t d = 1; d < 32; d <<= 1) {
            const unsigned long long y = __shfl_up_sync(kFull, x, d);
            if (lane >= d) x += y;
        }
        if (lane == 31) s_w[warp] = x;
        __syncthreads();
        unsigned long long before = from;
        for (uint32_t w = 0; w < kBW; ++w) {
            if (w < warp) before += s_w[w];
            from += s_w[w];
        }
        __syncthreads();
        return before + x - v;
    };
    for (uint32_t k = 0; k < kPlacePer; ++k) {
        const uint32_t p = blockIdx.x * kPlace + k * 256 + threadIdx.x;
        const bool on = p < n;
        PolyMeta m{};
        if (on) m = meta[p];
        const unsigned long long slot_off = scan(on ? poly_slots(m) : 0ull, base);
        uint32_t path = kPaths, records = 0;
        if (on) {
            m.slot_off = slot_off;
            path = m.err ? (uint32_t)kPaths : path_of(m, g, off[p + 1] - off[p], gain, records);
        }
        for (uint32_t q = 0; q < kPaths; ++q) {  // the lists (one add a warp)
            const uint32_t mask = __ballot_sync(kFull, path == q);
            if (!mask || q == kTiled) continue;
            uint32_t pos = 0;
            if (lane == __ffs(mask) - 1u) pos = atomicAdd(&tot->count[q], (uint32_t)__popc(mask));
            pos = __shfl_sync(kFull, pos, __ffs(mask) - 1) + __popc(mask & ((1u << lane) - 1u));
            if (path == q) lists[(uint64_t)q * n + pos] = p;
        }
        if (path == kTiled) {  // list place and first record by one add, so that both rise together
            const unsigned long long a = atomicAdd(&tot->tiled, 1ull << 40 | records);
            lists[(uint64_t)kTiled * n + (uint32_t)(a >> 40)] = p;
            m.item_off = (uint32_t)(a & ((1ull << 40) - 1));
        } else if (path == kSorted) {
            const CellWin W = window_of(m.mbr, g);
            m.rb_off = atomicAdd(&tot->srb, (unsigned long long)(W.wj1 - W.wj0 + 2));
        }
        if (__syncthreads_or(path == kSorted)) {
            const unsigned long long key_off = scan(path == kSorted ? m.T : 0u, kbase),
                                     cross_off = scan(path == kSorted ? m.inc : 0u, cbase);
            if (path == kSorted) m.key_off = key_off, m.cross_off = cross_off;
        }
        if (on) meta[p] = m;
    }
}

// ----------------------------------------------------------------- raster
// A window of H rows of 32 * WW cells (from column x0, row y0, multiples of 8)
// as bitmaps in shared memory, rows PITCH words apart (odd: the rows of a
// warp's threads fall in different banks).
template <uint32_t NT>
struct Raster {
    static constexpr uint32_t WW = NT == 32 ? 2 : 8, PITCH = WW + 1, H = NT == 32 ? 64 : 256;
    uint32_t a[H * PITCH];   // cells touched, then A
    uint32_t f[H * PITCH];   // cells entered, then F
    uint32_t x[H * PITCH];   // the turns
    uint32_t left[H / 32 + 1];  // bit r: the turns of the edges left of the window differ between rows r - 1 and r
    WalkShared<NT> walk;
};

// Sets bits [i0, i1] of a row.
__device__ __forceinline__ void set_bits(uint32_t *row, uint32_t i0, uint32_t i1) {
    for (uint32_t w = i0 >> 5; w <= i1 >> 5; ++w) {
        const uint32_t lo = w == i0 >> 5 ? i0 & 31u : 0u, hi = w == i1 >> 5 ? i1 & 31u : 31u;
        atomicOr(row + w, (0xffffffffu << lo) & (0xffffffffu >> (31u - hi)));
    }
}

// Rasters the polygon's cells of the window: A and F bitmaps in R.a and R.f.
template <uint32_t NT>
__device__ __forceinline__ void raster_window(const int2 *__restrict__ xy, uint64_t b, uint64_t nv, const GridP &g,
                                              int l, int32_t x0, int32_t y0, uint32_t rows, Raster<NT> &R) {
    using RT = Raster<NT>;
    const uint32_t t = Team<NT>::rank();
    for (uint32_t k = t; k < rows * RT::PITCH; k += NT) R.a[k] = R.f[k] = R.x[k] = 0;
    for (uint32_t k = t; k < RT::H / 32 + 1; k += NT) R.left[k] = 0;
    Team<NT>::sync();
    const int32_t x1 = min(x0 + 32 * (int32_t)RT::WW, (int32_t)g.G) - 1, y1 = min(y0 + (int32_t)rows, (int32_t)g.G) - 1;
    const int32_t xl = x0 << l, xr = (x1 + 1) << l;
    walk_edges<NT>(
        xy, b, nv, 0, nv, g, l, y0, y1, R.walk,
        [&](const EdgeRel &e) {
            if (min(e.ax, e.bx) > xr) return false;
            if (max(e.ax, e.bx) >= xl) return true;
            // left of the window: it turns every cell of the rows whose centre lines it crosses
            int32_t r0, r1;
            rel_centre_rows(e, l, r0, r1);
            r0 = max(r0, y0) - y0, r1 = min(r1, y1) - y0;
            if (r1 >= r0) {
                atomicXor(R.left + (r0 >> 5), 1u << (r0 & 31));
                atomicXor(R.left + ((r1 + 1) >> 5), 1u << ((r1 + 1) & 31));
            }
            return false;
        },
        [&](const RowCells &c) {
            const uint32_t row = (uint32_t)(c.j - y0) * RT::PITCH;
            const int32_t i0 = max(c.i0, x0), i1 = min(c.i1, x1), c0 = max(c.c0, x0), c1 = min(c.c1, x1);
            if (i1 >= i0) set_bits(R.a + row, (uint32_t)(i0 - x0), (uint32_t)(i1 - x0));
            if (c1 >= c0) set_bits(R.f + row, (uint32_t)(c0 - x0), (uint32_t)(c1 - x0));
            if (c.turns && c.t <= x1) {
                const uint32_t i = (uint32_t)(max(c.t, x0) - x0);
                atomicXor(R.x + row + (i >> 5), 1u << (i & 31u));
            }
        });
    // a prefix XOR along the row: the cells whose centre lies inside
    for (uint32_t r = t; r < rows; r += NT) {
        uint32_t par = 0;
        for (uint32_t w = 0; w < (r >> 5); ++w) par ^= R.left[w];
        par = __popc(par) + __popc(R.left[r >> 5] & (0xffffffffu >> (31u - (r & 31u))));
        uint32_t in = par & 1u ? 0xffffffffu : 0u;
#pragma unroll
        for (uint32_t w = 0; w < RT::WW; ++w) {
            const uint32_t k = r * RT::PITCH + w;
            uint32_t v = R.x[k];
            v ^= v << 1;
            v ^= v << 2;
            v ^= v << 4;
            v ^= v << 8;
            v ^= v << 16;
            v ^= in;
            in = v >> 31 ? 0xffffffffu : 0u;
            const int32_t past = x0 + 32 * (int32_t)w + 31 - x1;  // columns of the word behind the grid
            if (past > 0) v = past >= 32 ? 0u : v & (0xffffffffu >> past);
            if (y0 + (int32_t)r > y1) v = 0;
            const uint32_t full = v & ~R.f[k];
            R.f[k] = full;
            R.a[k] |= full;
        }
    }
    Team<NT>::sync();
}

// The table of hilbert_rows, in shared memory.
constexpr uint32_t kTabSize = 4 * 2 * 256;
struct TabRef {
    const uint16_t *e;
    __device__ __forceinline__ uint32_t operator()(uint32_t s, uint32_t half, uint32_t c) const {
        return e[(s * 2 + half) * 256 + c];
    }
};

// The squares of blocks a scan runs over, in Hilbert order.
struct Squares {
    uint32_t id[32], state[32];
    int32_t x[32], y[32];  // their first blocks
    uint32_t n;
};

// Fills the squares of cover c on a curve of `levels` block levels: lane k of
// a warp takes square k and its place from the ids below its own.
__device__ __forceinline__ void make_squares(const Cover &c, uint32_t levels, Squares &sq) {
    const uint32_t k = threadIdx.x & 31u;
    const bool on = k < c.n;
    const uint32_t x = (uint32_t)(c.x0 >> c.m) + k % c.nx, y = (uint32_t)(c.y0 >> c.m) + k / c.nx;
    uint32_t s = 0;
    const uint32_t id = on ? hilbert_id_state(levels - c.m, x, y, s) : 0xffffffffu;
    uint32_t at = 0;
    for (uint32_t j = 0; j < c.n; ++j) at += __shfl_sync(kFull, id, (int)j) < id ? 1u : 0u;
    if (on) sq.id[at] = id, sq.state[at] = s, sq.x[at] = (int32_t)(x << c.m), sq.y[at] = (int32_t)(y << c.m);
    if (k == 0) sq.n = c.n;
}

// A thread's run of PER blocks that follow each other on the curve, as the
// bits of their 64 cells in order, for A and F.
template <uint32_t PER>
struct BlockRun {
    uint64_t a[PER], f[PER];
    uint32_t id;  // of the first block
};

// Loads the run of blocks from position p of the squares on (4^m blocks each)
// out of the bitmaps (whose first block is (ox, oy)); blocks outside
// [bx0, bx1] x [by0, by1] and positions behind the squares are empty.
template <uint32_t NT, uint32_t PER>
__device__ __forceinline__ void load_run(const Raster<NT> &R, const TabRef &tab, const Squares &sq, uint32_t m,
                                         int32_t ox, int32_t oy, int32_t bx0, int32_t by0, int32_t bx1, int32_t by1,
                                         uint32_t p, BlockRun<PER> &run) {
    using RT = Raster<NT>;
    static_assert(PER == 1 || PER == 4, "a run is a block or the four of a square");
#pragma unroll
    for (uint32_t k = 0; k < PER; ++k) run.a[k] = run.f[k] = 0;
    run.id = 0;
    const uint32_t q = p >> (2 * m);
    if (q >= sq.n) return;
    const uint32_t d = p & ((1u << (2 * m)) - 1);
    run.id = sq.id[q] << (2 * m) | d;
    const uint32_t up = PER == 4 && m ? 1u : 0u;  // the levels below the run's square
    uint32_t s = sq.state[q], x, y;
    hilbert_square(m - up, d >> (2 * up), s, x, y);
    const int32_t X = sq.x[q] + (int32_t)(x << up), Y = sq.y[q] + (int32_t)(y << up);
    if (X + (int32_t)up < bx0 || Y + (int32_t)up < by0 || X > bx1 || Y > by1) return;
#pragma unroll
    for (uint32_t k = 0; k < PER; ++k) {
        int32_t bx = X, by = Y;
        uint32_t t = s;
        if (PER == 4 && up) {
            uint32_t cx = k >> 1, cy = (k >> 1) ^ (k & 1u);
            apply_sym(s, cx, cy);
            t ^= k == 0 ? 1u : k == 3 ? 2u : 0u;
            bx += (int32_t)cx, by += (int32_t)cy;
        } else if (k) {
            break;  // the only block of a square without levels
        }
        if (bx < bx0 || by < by0 || bx > bx1 || by > by1) continue;
        const uint8_t *pa = (const uint8_t *)(R.a + 8 * (by - oy) * (int32_t)RT::PITCH) + (bx - ox);
        const uint8_t *pf = (const uint8_t *)(R.f + 8 * (by - oy) * (int32_t)RT::PITCH) + (bx - ox);
        constexpr uint32_t P = RT::PITCH * 4;
        const uint32_t a0 = pa[0] | pa[P] << 8 | pa[2 * P] << 16 | (uint32_t)pa[3 * P] << 24;
        const uint32_t a1 = pa[4 * P] | pa[5 * P] << 8 | pa[6 * P] << 16 | (uint32_t)pa[7 * P] << 24;
        if (!(a0 | a1)) continue;  // F is a part of A
        const uint32_t f0 = pf[0] | pf[P] << 8 | pf[2 * P] << 16 | (uint32_t)pf[3 * P] << 24;
        const uint32_t f1 = pf[4 * P] | pf[5 * P] << 8 | pf[6 * P] << 16 | (uint32_t)pf[7 * P] << 24;
        run.a[k] = (a0 & a1) == 0xffffffffu ? ~0ull : block_in_order(tab, t, a0, a1);
        run.f[k] = (f0 & f1) == 0xffffffffu ? ~0ull : (f0 | f1) ? block_in_order(tab, t, f0, f1) : 0ull;
    }
}

// The interval starts of a run whose predecessor cell's bit is prev.
template <uint32_t PER>
__device__ __forceinline__ uint32_t run_starts(const uint64_t (&w)[PER], uint32_t prev) {
    uint32_t n = 0;
#pragma unroll
    for (uint32_t k = 0; k < PER; ++k) {
        n += (uint32_t)__popcll(w[k] & ~(w[k] << 1 | prev));
        prev = (uint32_t)(w[k] >> 63);
    }
    return n;
}

// Writes a run's intervals: a cell in the list whose predecessor is not starts
// one (its id to x), a cell not in it whose predecessor is ends it (to y).
// `start` intervals have started before the run; `close` ends one that
// reaches the run's end there.
template <uint32_t PER>
__device__ __forceinline__ void write_run(const uint64_t (&w)[PER], uint32_t prev, uint32_t id, uint32_t blocks,
                                          uint32_t start, bool close, uint2 *out) {
    uint32_t i = start, k = start - prev;
#pragma unroll
    for (uint32_t b = 0; b < PER; ++b) {
        if (b >= blocks) break;
        const uint32_t c = (id + b) << 6;
        for (uint64_t e = ~w[b] & (w[b] << 1 | prev); e; e &= e - 1)
            out[k++].y = c + (uint32_t)__ffsll((long long)e) - 1u;
        for (uint64_t e = w[b] & ~(w[b] << 1 | prev); e; e &= e - 1)
            out[i++].x = c + (uint32_t)__ffsll((long long)e) - 1u;
        prev = (uint32_t)(w[b] >> 63);
    }
    if (close && prev) out[k].y = (id + blocks) << 6;  // 2^32 wraps to 0 by design
}

// The last cells' bits (A, F << 1) of the run before each thread's; thread 0
// gets `carry`, and *last the bits of the team's last run.
template <uint32_t NT>
__device__ __forceinline__ uint32_t bits_before(uint32_t mine, uint32_t carry, uint32_t &last, uint32_t *sums) {
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    uint32_t v = __shfl_up_sync(kFull, mine, 1);
    if (NT == 32) {
        last = __shfl_sync(kFull, mine, 31);
        return lane ? v : carry;
    }
    if (lane == 31) sums[16 + warp] = mine;
    __syncthreads();
    if (lane == 0) v = warp ? sums[15 + warp] : carry;
    last = sums[16 + NT / 32 - 1];
    __syncthreads();
    return v;
}

// Reads a whole window's bitmaps back in Hilbert order and writes its lists;
// returns their lengths.
template <uint32_t NT, uint32_t PER>
__device__ __forceinline__ uint2 scan_window(const Raster<NT> &R, const TabRef &tab, const Squares &sq, uint32_t m,
                                             int32_t bx0, int32_t by0, int32_t bx1, int32_t by1, uint2 *Aout,
                                             uint2 *Fout, uint32_t *sums) {
    const uint32_t per = 1u << (2 * m), total = sq.n << (2 * m), t = Team<NT>::rank();
    uint32_t na = 0, nf = 0, carry = 0;
    for (uint32_t p0 = 0; p0 < total; p0 += NT * PER) {
        const uint32_t p = p0 + t * PER, q = p >> (2 * m), d = p & (per - 1);
        BlockRun<PER> run;
        load_run<NT, PER>(R, tab, sq, m, bx0, by0, bx0, by0, bx1, by1, p, run);
        const uint32_t blocks = min((uint32_t)PER, per);
        const uint32_t mine = (uint32_t)(run.a[PER - 1] >> 63) | (uint32_t)(run.f[PER - 1] >> 63) << 1;
        uint32_t last;
        uint32_t prev = bits_before<NT>(mine, carry, last, sums);
        carry = last;
        const bool on = q < sq.n;
        if (on && d == 0 && q > 0 && sq.id[q] != sq.id[q - 1] + 1u) prev = 0;  // a gap of the curve
        if (!on) prev = 0;
        uint32_t all;  // 1,024 blocks hold at most 2^15 starts: 16 bits each
        const uint32_t ex = Team<NT>::scan(run_starts(run.a, prev & 1u) | run_starts(run.f, prev >> 1) << 16, all, sums);
        if (on) {
            const bool close = d + blocks == per && !(q + 1 < sq.n && sq.id[q + 1] == sq.id[q] + 1u);
            write_run(run.a, prev & 1u, run.id, blocks, na + (ex & 0xffffu), close, Aout);
            write_run(run.f, prev >> 1, run.id, blocks, nf + (ex >> 16), close, Fout);
        }
        na += all & 0xffffu;
        nf += all >> 16;
    }
    return make_uint2(na, nf);
}

// The levels of the curve the blocks are numbered on: grids of fewer than
// 8 x 8 cells sit in the corner of one two levels larger, which visits them
// first and in the same order.
__device__ __forceinline__ uint32_t curve_order(uint32_t order) { return order < 3 ? order + 2 : order; }

// A polygon whose window one raster holds.
template <uint32_t NT>
__device__ __forceinline__ void build_window(const int2 *__restrict__ xy, const uint64_t *__restrict__ off, uint32_t p,
                                             const PolyMeta &M, const GridP &g, int l, Raster<NT> &R, Squares &sq,
                                             const TabRef &tab, uint32_t *sums, uint32_t *desc_out, int4 *mbr_out,
                                             uint2 *iv_out) {
    const uint32_t t = Team<NT>::rank();
    const uint64_t f_off = M.slot_off + even_up((uint64_t)M.T + 1);
    uint2 len = make_uint2(1, 1);
    if (M.T == 0) {  // it holds the whole grid (the count checked)
        if (t == 0) {
            const uint32_t cells = (uint32_t)((uint64_t)g.G * (uint64_t)g.G);  // 2^32 wraps to 0 by design
            iv_out[M.slot_off] = iv_out[f_off] = make_uint2(0u, cells);
        }
    } else {
        const CellWin W = window_of(M.mbr, g);
        const Cover c = cover_of(W, 3);
        if (t < 32) make_squares(c, curve_order(g.order) - 3, sq);
        raster_window<NT>(xy, off[p], off[p + 1] - off[p], g, l, 8 * c.x0, 8 * c.y0, 8u * (uint32_t)(c.y1 - c.y0 + 1), R);
        // small windows have a few blocks for each lane to share, larger ones
        // enough for every thread to take four in a row
        len = scan_window<NT, NT == 32 ? 1 : 4>(R, tab, sq, c.m, c.x0, c.y0, c.x1, c.y1, iv_out + M.slot_off,
                                                iv_out + f_off, sums);
    }
    if (t == 0) {
        ((uint4 *)desc_out)[p] = make_uint4((uint32_t)M.slot_off, len.x, (uint32_t)f_off, len.y);
        mbr_out[p] = make_int4(M.mbr[0], M.mbr[1], M.mbr[2], M.mbr[3]);
    }
    Team<NT>::sync();
}

// Fills the table (2 KB entries made of two nibbles: a cell at a time, so that
// each thread walks 16 positions for its own entries only).
__device__ __forceinline__ void load_tab(uint16_t *tab) {
    for (uint32_t k = threadIdx.x; k < kTabSize; k += blockDim.x) tab[k] = hilbert_rows(k >> 9, k >> 8 & 1u, k & 255u);
    __syncthreads();
}

// Windows up to 64 x 64 cells, a warp each: most of a layer's polygons, whose
// edges would leave a CTA's threads idle.  Bound by issue (the row walk and
// the scan of the blocks); 1.3 ms of 200,000 layer polygons' 9.6.  Emitting,
// sorting and scanning their cells instead took 66.5 ms for the layer.
__global__ void __launch_bounds__(256) k_bsmall(const int2 *__restrict__ xy, const uint64_t *__restrict__ off,
                                                const uint32_t *__restrict__ list, uint32_t n, GridP g, int l,
                                                const PolyMeta *__restrict__ meta, uint32_t *desc_out, int4 *mbr_out, uint2 *iv_out) {
    __shared__ Raster<32> R[kBW];
    __shared__ Squares sq[kBW];
    __shared__ uint16_t tab[kTabSize];
    load_tab(tab);
    const uint32_t warp = threadIdx.x >> 5;
    for (uint32_t q = blockIdx.x * kBW + warp; q < n; q += gridDim.x * kBW) {
        const uint32_t p = list[q];
        build_window<32>(xy, off, p, meta[p], g, l, R[warp], sq[warp], TabRef{tab}, nullptr, desc_out, mbr_out, iv_out);
    }
}

// Windows up to 256 x 256 cells, a CTA each.  Bound by issue and by the
// barriers between its steps, which other CTAs of the SM fill; 2.4 ms of
// 200,000 layer polygons' 9.6.
// CTAs per SM the 256-thread raster kernels are compiled for (shared memory
// holds six): with three the layer took a tenth longer than with four, with
// five 9.8 ms instead of 9.65.
#ifndef APRIL_RASTER_BLOCKS
#define APRIL_RASTER_BLOCKS 4
#endif
__global__ void __launch_bounds__(256, APRIL_RASTER_BLOCKS)
    k_bmid(const int2 *__restrict__ xy, const uint64_t *__restrict__ off, const uint32_t *__restrict__ list, uint32_t n,
           GridP g, int l, const PolyMeta *__restrict__ meta, uint32_t *desc_out, int4 *mbr_out, uint2 *iv_out) {
    __shared__ Raster<256> R;
    __shared__ Squares sq;
    __shared__ uint32_t sums[32];
    __shared__ uint16_t tab[kTabSize];
    load_tab(tab);
    for (uint32_t q = blockIdx.x; q < n; q += gridDim.x) {
        const uint32_t p = list[q];
        build_window<256>(xy, off, p, meta[p], g, l, R, sq, TabRef{tab}, sums, desc_out, mbr_out, iv_out);
    }
}

// ------------------------------------------------------------------- tiles
// Tile records, in each polygon's Hilbert order of the squares of its tile
// cover (tiles outside the window included).  A tile's CTA publishes the
// interval starts it counts by itself with its first and last cells' bits
// (own), then, once it has found the starts before it, the starts up to its
// end (upto).  Each word says in its top bit that it is there.
struct TileRec {
    unsigned long long own;   // na << 8 | nf << 32 | first A, first F, last A, last F in bits 0 to 3
    unsigned long long upto;  // na | nf << 31, or kFailed
};
constexpr unsigned long long kThere = 1ull << 63;
constexpr unsigned long long kFailed = 1ull << 62;  // upto: the tile's look-back ran out
constexpr uint32_t kTileFailed = 5;                 // PolyMeta.err: one of its tiles' did

__device__ __forceinline__ unsigned long long peek(const unsigned long long *p) {
    return *(const volatile unsigned long long *)p;
}

// The starts before record `it` of a polygon whose first record is `first`,
// and the last cells' bits of the record before it, by one warp: 32 records
// at a time back to the nearest known prefix.  joined(k) says whether record k
// follows k - 1 on the curve.  Records are handed out in order, so the ones
// waited for belong to CTAs that run; the wait is bounded all the same (at
// most c_tile_spins polls a step, lowered by the diagnostic wait limit), and
// false says that it ran out, here or in a tile whose sum this one needs.
constexpr uint32_t kTileSpins = 1u << 22;
__constant__ uint32_t c_tile_spins = kTileSpins;
template <class Joined>
__device__ __forceinline__ bool starts_before(const TileRec *recs, uint32_t it, uint32_t first, Joined joined,
                                              uint32_t &na, uint32_t &nf, uint32_t &prev) {
    const uint32_t lane = threadIdx.x & 31u;
    na = nf = prev = 0;
    if (it == first) return true;
    uint32_t end = it;  // records [first, end) are still to be summed up
    for (;;) {
        const bool on = lane < end - first;
        const uint32_t k = end - 1u - lane;  // lane 0 has the nearest
        unsigned long long own = 0, upto = 0;
        uint32_t known = 0, have = 0;
        for (uint32_t spin = 0;; ++spin) {
            if (spin == c_tile_spins) return false;
            if (on) {
                upto = peek(&recs[k].upto);
                own = peek(&recs[k].own);
            }
            have = __ballot_sync(kFull, !on || (own & kThere));
            known = __ballot_sync(kFull, on && (upto & kThere));
            const uint32_t need = known ? (2u << (__ffs(known) - 1)) - 1u : kFull;  // up to the nearest prefix
            if ((have & need) == need) break;
        }
        if (end == it) {
            const uint32_t bits = __shfl_sync(kFull, (uint32_t)own & 15u, 0);
            prev = joined(it) ? bits >> 2 : 0u;
        }
        // record k's starts, less those its predecessor's last cell already began
        const uint32_t last = __shfl_down_sync(kFull, (uint32_t)own >> 2 & 3u, 1);
        const uint32_t sub = on && k > first && joined(k) ? (uint32_t)own & last : 0u;
        const uint32_t stop = known ? (uint32_t)__ffs(known) - 1u : 31u;  // lanes before it count their own
        uint32_t a = 0, f = 0;
        if (on && lane < stop) {
            a = ((uint32_t)(own >> 8) & 0xffffffu) - (sub & 1u);
            f = ((uint32_t)(own >> 32) & 0xffffffu) - (sub >> 1 & 1u);
        }
        na += __reduce_add_sync(kFull, a);
        nf += __reduce_add_sync(kFull, f);
        if (known) {
            const unsigned long long u = __shfl_sync(kFull, upto, (int)stop);
            if (u & kFailed) return false;
            na += (uint32_t)u & 0x7fffffffu;
            nf += (uint32_t)(u >> 31) & 0x7fffffffu;
            return true;
        }
        // lane 31's own starts wait for its predecessor's bits: the next step takes it
        if (end - first <= 31u) return true;
        end -= 31u;
    }
}

// Empties the records, with each one's polygon in its own word; a warp per polygon.
__global__ void __launch_bounds__(256) k_btinit(const uint32_t *__restrict__ list, uint32_t n, GridP g,
                                                const PolyMeta *__restrict__ meta, TileRec *recs) {
    for (uint32_t i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n; i += gridDim.x * kBW) {
        const uint32_t p = list[i], first = meta[p].item_off;
        const Cover c = cover_of(window_of(meta[p].mbr, g), 8);
        for (uint32_t k = threadIdx.x & 31u; k < c.n << (2 * c.m); k += 32) recs[first + k] = TileRec{p, 0};
    }
}

// A tile of 256 x 256 cells a CTA, in order, from a counter, so that the
// earlier tiles a look-back waits for have been started.  One pass over the
// tiles: counting, summing and writing in three cost 12 ms of the layer's 18.8,
// this 3.9 of its 9.6, and 2.2 of the 2.9 that 1,000 query polygons of 540
// vertices take (47 when their cells were sorted).  Each tile walks all edges
// of its polygon, most of which miss it.  A tile whose look-back runs out
// writes no intervals; its polygon's lists then end up empty, and the context's
// status says so.
__global__ void __launch_bounds__(256, APRIL_RASTER_BLOCKS)
    k_btile(const int2 *__restrict__ xy, const uint64_t *__restrict__ off, uint32_t items, GridP g, int l,
            PolyMeta *meta, TileRec *recs, uint32_t *counter, uint32_t *status, uint32_t *desc_out, int4 *mbr_out,
            uint2 *iv_out) {
    __shared__ Raster<256> R;
    __shared__ Squares tsq, sq;
    __shared__ uint32_t sums[32];
    __shared__ uint16_t tab[kTabSize];
    __shared__ uint32_t s_item, s_before[4];
    load_tab(tab);
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(counter, 1u);
        __syncthreads();
        const uint32_t it = s_item;
        if (it >= items) break;
        const uint32_t p = (uint32_t)peek(&recs[it].own);  // k_btinit left the polygon here
        const PolyMeta M = meta[p];
        const CellWin W = window_of(M.mbr, g);
        const Cover c = cover_of(W, 8);
        if (threadIdx.x < 32) make_squares(c, g.order - 8, tsq);
        __syncthreads();
        const uint32_t per = 1u << (2 * c.m), total = c.n << (2 * c.m);
        // the tile at place q of the polygon's records, and whether the window holds it
        auto tile_at = [&](uint32_t q, uint32_t &s, int32_t &tx, int32_t &ty) {
            const uint32_t sqi = q >> (2 * c.m);
            uint32_t x, y;
            s = tsq.state[sqi];
            hilbert_square(c.m, q & (per - 1), s, x, y);
            tx = tsq.x[sqi] + (int32_t)x, ty = tsq.y[sqi] + (int32_t)y;
            return tx >= c.x0 && tx <= c.x1 && ty >= c.y0 && ty <= c.y1;
        };
        auto joined = [&](uint32_t rec) {  // record rec follows the one before it on the curve
            const uint32_t q = rec - M.item_off, sqi = q >> (2 * c.m);
            return (q & (per - 1)) || (sqi && tsq.id[sqi] == tsq.id[sqi - 1] + 1u);
        };
        const uint32_t q = it - M.item_off;
        uint32_t s;
        int32_t tx, ty;
        const bool in = tile_at(q, s, tx, ty);
        BlockRun<4> run{};
        uint32_t last = 0;
        if (in) {
            if (threadIdx.x == 0) {
                sq.n = 1;
                sq.id[0] = tsq.id[q >> (2 * c.m)] << (2 * c.m) | (q & (per - 1));
                sq.state[0] = s;
                sq.x[0] = 32 * tx;
                sq.y[0] = 32 * ty;
            }
            // the window's part of the tile
            const int32_t bx0 = max(32 * tx, (int32_t)(W.wi0 >> 3)), bx1 = min(32 * tx + 31, (int32_t)(W.wi1 >> 3));
            const int32_t by0 = max(32 * ty, (int32_t)(W.wj0 >> 3)), by1 = min(32 * ty + 31, (int32_t)(W.wj1 >> 3));
            raster_window<256>(xy, off[p], off[p + 1] - off[p], g, l, 256 * tx, 8 * by0, 8u * (uint32_t)(by1 - by0 + 1), R);
            load_run<256, 4>(R, TabRef{tab}, sq, 5u, 32 * tx, by0, bx0, by0, bx1, by1, 4 * threadIdx.x, run);
        }
        const uint32_t mine = (uint32_t)(run.a[3] >> 63) | (uint32_t)(run.f[3] >> 63) << 1;
        uint32_t before = bits_before<256>(mine, 0u, last, sums);
        uint32_t all;
        Team<256>::scan(run_starts(run.a, before & 1u) | run_starts(run.f, before >> 1) << 16, all, sums);
        if (threadIdx.x == 0) {
            const uint32_t first = (uint32_t)(run.a[0] & 1u) | (uint32_t)(run.f[0] & 1u) << 1;
            *(volatile unsigned long long *)&recs[it].own = kThere | (unsigned long long)(all & 0xffffu) << 8 |
                                                            (unsigned long long)(all >> 16) << 32 | first | last << 2;
            s_before[3] = first;
        }
        if (!in && q + 1 < total) {  // nothing to write, and its neighbours sum up past it
            __syncthreads();
            continue;
        }
        if (threadIdx.x < 32) {
            uint32_t na, nf, prev;
            const bool ok = starts_before(recs, it, M.item_off, joined, na, nf, prev);
            if (threadIdx.x == 0) {
                const uint32_t sub = prev & s_before[3];
                const unsigned long long ua = na + (all & 0xffffu) - (sub & 1u), uf = nf + (all >> 16) - (sub >> 1);
                *(volatile unsigned long long *)&recs[it].upto = kThere | (ok ? ua | uf << 31 : kFailed);
                s_before[0] = na, s_before[1] = nf, s_before[2] = ok ? prev : 4u;
                auto put = [&](uint32_t la, uint32_t lf) {
                    ((uint4 *)desc_out)[p] = make_uint4((uint32_t)M.slot_off, la,
                                                        (uint32_t)(M.slot_off + even_up((uint64_t)M.T + 1)), lf);
                };
                // the last tile gives the lengths, 0 where some tile failed: a tile that fails marks the
                // polygon before it writes 0, the last one looks for the mark after it wrote the lengths
                volatile uint32_t *err = &meta[p].err;
                if (!ok) {
                    atomicOr(status, kStatusTimeout);
                    *err = kTileFailed;
                    __threadfence();
                } else if (q + 1 == total) {
                    put((uint32_t)ua, (uint32_t)uf);
                    __threadfence();
                }
                if (!ok || (q + 1 == total && *err)) put(0u, 0u);
                if (q + 1 == total) mbr_out[p] = make_int4(M.mbr[0], M.mbr[1], M.mbr[2], M.mbr[3]);
            }
        }
        __syncthreads();
        const uint32_t prev = s_before[2];
        if (in && prev < 4u) {
            if (threadIdx.x == 0) before = prev;
            const uint32_t ex = Team<256>::scan(
                run_starts(run.a, before & 1u) | run_starts(run.f, before >> 1) << 16, all, sums);
            // the last run ends an interval that the next record does not go on with
            uint32_t s1;
            int32_t x1, y1;
            const bool close = threadIdx.x == 255 &&
                               !(q + 1 < total && joined(it + 1) && tile_at(q + 1, s1, x1, y1));
            write_run(run.a, before & 1u, run.id, 4u, s_before[0] + (ex & 0xffffu), close, iv_out + M.slot_off);
            write_run(run.f, before >> 1, run.id, 4u, s_before[1] + (ex >> 16), close,
                      iv_out + M.slot_off + even_up((uint64_t)M.T + 1));
        }
        __syncthreads();
    }
}

// ------------------------------------------- CTA helpers (sorted path)
struct BuildShared {
    uint32_t warp_sum[kBW];
    uint32_t item;
    uint32_t k_count;
};

// Exclusive scan of one value per thread over the CTA; *total gets the sum.
__device__ __forceinline__ uint32_t block_scan(uint32_t v, uint32_t &total, BuildShared &sh) {
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    uint32_t x = v;
    for (uint32_t d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, x, d);
        if (lane >= d) x += y;
    }
    if (lane == 31) sh.warp_sum[warp] = x;
    __syncthreads();
    uint32_t before = 0, all = 0;
    for (uint32_t w = 0; w < kBW; ++w) {
        if (w < warp) before += sh.warp_sum[w];
        all += sh.warp_sum[w];
    }
    __syncthreads();
    total = all;
    return before + x - v;
}


// Point-in-polygon at the centre of cell (i, j), the host builder's rule: an
// upward edge toggles when the centre is strictly left of it, i.e. when its
// crossing x is greater than the centre's.  The centre is never on the
// boundary here (it lies in the open square of a cell the boundary does not
// enter), so x > xc is floor(x) >= xc, and the parity of the row's sorted
// crossings at or right of xc decides.  Cells outside the window are outside.
__device__ bool inside_cell(uint32_t i, uint32_t j, const PolyMeta &M, const CellWin &W, const GridP &g,
                            const uint32_t *row_start, const unsigned long long *cross) {
    if ((int64_t)i < W.wi0 || (int64_t)i > W.wi1 || (int64_t)j < W.wj0 || (int64_t)j > W.wj1) return false;
    const int64_t xc = g.ox + (int64_t)i * g.h + g.h / 2;
    const uint32_t r = j - (uint32_t)W.wj0;
    uint32_t lo = row_start[r];
    const uint32_t hi = row_start[r + 1];
    const int64_t xr = xc - M.mbr[0];
    if (xr > 0) {
        const unsigned long long xk = (unsigned long long)imin(xr, (1ll << kCrossXBits) - 1);
        uint32_t h2 = hi;
        while (lo < h2) {  // first crossing with floor(x) - xmn >= xc - xmn
            const uint32_t mid = (lo + h2) >> 1;
            if ((cross[mid] & ((1ull << kCrossXBits) - 1)) < xk) lo = mid + 1;
            else h2 = mid;
        }
    }
    return ((hi - lo) & 1u) != 0;
}

// ------------------------------------- (edge, row) work items (sorted path)
// The closed strips of cell rows an edge meets, flattened over a polygon's
// edges so that the CTA's threads share them evenly whatever the edges'
// lengths.  Edges are taken kChunkE at a time; for a chunk, pre[e] is the
// number of items before local edge e and j0[e] its first row.
constexpr uint32_t kChunkE = 1024;
struct EdgeChunk {
    uint32_t pre[kChunkE + 1];
    int32_t j0[kChunkE];
};

// Fills the chunk of edges [e_base, e_base + ne) and returns its item count.
__device__ uint32_t load_chunk(const int2 *xy, uint64_t b, uint64_t nv, uint64_t e_base, uint32_t ne, const GridP &g,
                               EdgeChunk &ch, BuildShared &sh) {
    constexpr uint32_t per = kChunkE / kBB;
    uint32_t cnt[per], sum = 0;
    for (uint32_t q = 0; q < per; ++q) {
        const uint32_t e = threadIdx.x * per + q;
        cnt[q] = 0;
        if (e < ne) {
            const int2 a = vtx(xy, b, nv, e_base + e), c = vtx(xy, b, nv, e_base + e + 1);
            int64_t j0, j1;
            edge_rows(edge_up(a.x, a.y, c.x, c.y), g.oy, g.h, g.G, j0, j1);
            ch.j0[e] = (int32_t)j0;
            cnt[q] = j1 >= j0 ? (uint32_t)(j1 - j0 + 1) : 0u;
        }
        sum += cnt[q];
    }
    uint32_t total;
    uint32_t run = block_scan(sum, total, sh);
    for (uint32_t q = 0; q < per; ++q) {
        const uint32_t e = threadIdx.x * per + q;
        if (e < kChunkE) ch.pre[e] = run;
        run += cnt[q];
    }
    if (threadIdx.x == 0) ch.pre[kChunkE] = total;
    __syncthreads();
    return total;
}

// The local edge of item q (the last e with pre[e] <= q) and its row.
__device__ __forceinline__ uint32_t item_edge(const EdgeChunk &ch, uint32_t ne, uint32_t q, int64_t &j) {
    uint32_t lo = 0, hi = ne - 1;
    while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) >> 1;
        if (ch.pre[mid] <= q) lo = mid;
        else hi = mid - 1;
    }
    j = ch.j0[lo] + (int64_t)(q - ch.pre[lo]);
    return lo;
}

// ------------------------------------------------------------------- sort
// Stable LSD radix sort of N 64-bit keys, 8 bits per pass.  A tile is 4096
// keys (256 threads x 16); per pass: k_rs_hist counts every tile's digits
// (digit-major table), k_rs_rows turns each digit's row into exclusive tile
// offsets and k_rs_digits the digit totals into digit bases, and
// k_rs_scatter moves every key to its digit base + tile offset + rank,
// ranking a tile's keys in order: 16 slices of 256, each ranked within its
// warp by match_any and across warps by per-warp digit counts.
constexpr unsigned kRsT = 256, kRsItems = 16, kRsTile = kRsT * kRsItems;

__global__ void __launch_bounds__(kRsT) k_rs_hist(const unsigned long long *__restrict__ src, uint64_t N,
                                                  uint32_t shift, uint32_t *hist, uint32_t ntiles) {
    __shared__ uint32_t h[256];
    const uint32_t tid = threadIdx.x;
    for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        h[tid] = 0;
        __syncthreads();
        for (uint32_t i = 0; i < kRsItems; ++i) {
            const uint64_t idx = (uint64_t)tile * kRsTile + i * kRsT + tid;
            if (idx < N) atomicAdd(&h[(uint32_t)(src[idx] >> shift) & 255u], 1u);
        }
        __syncthreads();
        hist[(uint64_t)tid * ntiles + tile] = h[tid];
        __syncthreads();
    }
}

constexpr unsigned kRsScanT = 1024;
__global__ void __launch_bounds__(kRsScanT) k_rs_rows(uint32_t *hist, uint32_t ntiles, uint32_t *totals) {
    __shared__ uint32_t s_w[kRsScanT / 32];
    uint32_t *row = hist + (uint64_t)blockIdx.x * ntiles;
    const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5;
    const uint32_t chunk = (ntiles + kRsScanT - 1) / kRsScanT;
    const uint32_t b = min(ntiles, t * chunk), e = min(ntiles, b + chunk);
    uint32_t sum = 0;
    for (uint32_t k = b; k < e; ++k) sum += row[k];
    uint32_t incl = sum;
    for (uint32_t d = 1; d < 32; d <<= 1) {
        const uint32_t v = __shfl_up_sync(kFull, incl, d);
        if (lane >= d) incl += v;
    }
    if (lane == 31) s_w[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = s_w[lane];
        for (uint32_t d = 1; d < 32; d <<= 1) {
            const uint32_t v = __shfl_up_sync(kFull, w, d);
            if (lane >= d) w += v;
        }
        s_w[lane] = w;
    }
    __syncthreads();
    uint32_t run = incl - sum + (warp ? s_w[warp - 1] : 0u);
    for (uint32_t k = b; k < e; ++k) {
        const uint32_t c = row[k];
        row[k] = run;
        run += c;
    }
    if (t == kRsScanT - 1) totals[blockIdx.x] = s_w[31];
}

__global__ void __launch_bounds__(256) k_rs_digits(uint32_t *totals) {
    __shared__ uint32_t v[256];
    const uint32_t t = threadIdx.x;
    v[t] = totals[t];
    __syncthreads();
    if (t == 0) {
        uint32_t run = 0;
        for (int d = 0; d < 256; ++d) {
            const uint32_t c = v[d];
            v[d] = run;
            run += c;
        }
    }
    __syncthreads();
    totals[t] = v[t];
}

__global__ void __launch_bounds__(kRsT) k_rs_scatter(const unsigned long long *__restrict__ src,
                                                     unsigned long long *__restrict__ dst, uint64_t N, uint32_t shift,
                                                     const uint32_t *__restrict__ hist,
                                                     const uint32_t *__restrict__ dbase, uint32_t ntiles) {
    __shared__ uint32_t run[256];
    __shared__ uint32_t wc[kRsT / 32][256];
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        run[tid] = dbase[tid] + hist[(uint64_t)tid * ntiles + tile];
        for (uint32_t w = 0; w < kRsT / 32; ++w) wc[w][tid] = 0;
        __syncthreads();
        for (uint32_t i = 0; i < kRsItems; ++i) {
            const uint64_t idx = (uint64_t)tile * kRsTile + i * kRsT + tid;
            const bool valid = idx < N;
            const unsigned long long key = valid ? src[idx] : 0ull;
            const uint32_t d = valid ? (uint32_t)(key >> shift) & 255u : 256u;
            const uint32_t peers = __match_any_sync(kFull, d);
            const uint32_t rank = __popc(peers & ((1u << lane) - 1u));
            if (valid && rank == 0) wc[warp][d] = __popc(peers);
            __syncthreads();
            {  // thread tid: the start of every warp's keys of digit tid
                uint32_t r = run[tid];
                for (uint32_t w = 0; w < kRsT / 32; ++w) {
                    const uint32_t c = wc[w][tid];
                    wc[w][tid] = r;
                    r += c;
                }
                run[tid] = r;
            }
            __syncthreads();
            if (valid) dst[wc[warp][d] + rank] = key;
            __syncthreads();
            for (uint32_t w = 0; w < kRsT / 32; ++w) wc[w][tid] = 0;
            __syncthreads();
        }
    }
}

// ------------------------------------------------------------------- emit
constexpr uint32_t kKeyBits = 33;  // Hilbert id (32 bits at order 16) << 1 | crossed
__global__ void __launch_bounds__(kBB) k_bemit(const int2 *__restrict__ xy, const uint64_t *__restrict__ off,
                                               const uint32_t *__restrict__ list, uint32_t n, GridP g,
                                               const PolyMeta *__restrict__ meta, unsigned long long *keys_all, unsigned long long *cross_all,
                                               uint32_t *counter) {
    __shared__ BuildShared sh;
    __shared__ EdgeChunk ch;
    const uint32_t tid = threadIdx.x;
    for (;;) {
        if (tid == 0) sh.item = atomicAdd(counter, 1u);
        __syncthreads();
        const uint32_t it = sh.item;
        __syncthreads();
        if (it >= n) break;
        const uint32_t p = list[it];
        const PolyMeta M = meta[p];
        const CellWin W = window_of(M.mbr, g);
        const uint64_t b = off[p], nv = off[p + 1] - b;
        const uint32_t T = M.T;  // a polygon with no touched cell still writes its crossings
        unsigned long long *keys = keys_all + M.key_off, *cross = cross_all + M.cross_off;
        const unsigned long long tag = (unsigned long long)p << kKeyBits;
        const unsigned long long ctag = (unsigned long long)p << kCrossPolyShift;
        uint32_t carry = 0, ccarry = 0;
        for (uint64_t e_base = 0; e_base < nv; e_base += kChunkE) {
            const uint32_t ne = (uint32_t)min((uint64_t)kChunkE, nv - e_base);
            const uint32_t R = load_chunk(xy, b, nv, e_base, ne, g, ch, sh);
            for (uint32_t q0 = 0; q0 < R; q0 += kBB) {
                const uint32_t q = q0 + tid;
                EdgeUp ed{0, 0, 0, 0};
                int64_t j = 0, i0 = 0, i1 = -1, r0 = 0, r1 = -1;
                if (q < R) {
                    const uint32_t e = item_edge(ch, ne, q, j);
                    const int2 a = vtx(xy, b, nv, e_base + e), c = vtx(xy, b, nv, e_base + e + 1);
                    ed = edge_up(a.x, a.y, c.x, c.y);
                    if (!edge_cells_in_row(ed, g.ox, g.oy, g.h, g.G, j, i0, i1)) i1 = i0 - 1;
                    centre_rows(ed, g.oy, g.h, W.wj0, W.wj1, r0, r1);
                }
                const bool crosses = q < R && j >= r0 && j <= r1;  // the edge crosses row j's centre line
                uint32_t total, ctotal;
                uint32_t pos = carry + block_scan(i1 >= i0 ? (uint32_t)(i1 - i0 + 1) : 0u, total, sh);
                const uint32_t cpos = ccarry + block_scan(crosses ? 1u : 0u, ctotal, sh);
                carry += total;
                ccarry += ctotal;
                const int64_t Y0 = g.oy + j * g.h;
                for (int64_t i = i0; i <= i1; ++i) {
                    const bool crossed = enters_open_square(ed.ax, ed.ay, ed.bx, ed.by, g.ox + i * g.h, Y0, g.h);
                    const unsigned long long key =
                        tag | (hilbert_id(g.order, (uint32_t)i, (uint32_t)j) << 1) | (crossed ? 1ull : 0ull);
                    if (pos < T) keys[pos] = key;
                    ++pos;
                }
                if (crosses && cpos < M.inc) {
                    const int64_t yc = Y0 + g.h / 2, den = ed.by - ed.ay;
                    const int64_t xf = floor_div(ed.ax * den + (yc - ed.ay) * (ed.bx - ed.ax), den);
                    cross[cpos] = ctag | ((unsigned long long)(j - W.wj0) << kCrossXBits) |
                                  (unsigned long long)(xf - M.mbr[0]);
                }
            }
            __syncthreads();
        }
    }
}

// ------------------------------------------------------------------ build
__global__ void __launch_bounds__(kBB) k_bconstruct(const int2 *__restrict__ xy, const uint64_t *__restrict__ off,
                                                    const uint32_t *__restrict__ list, uint32_t n, GridP g,
                                                    const PolyMeta *__restrict__ meta,
                                                    const unsigned long long *sorted_all, unsigned long long *other_all,
                                                    const unsigned long long *cross_all, uint8_t *flags_all,
                                                    uint32_t *rb_all, uint32_t *desc_out,
                                                    int4 *mbr_out, uint2 *iv_out, uint32_t *counter) {
    __shared__ BuildShared sh;
    const uint32_t tid = threadIdx.x;
    const uint64_t ncells = (uint64_t)g.G * (uint64_t)g.G;
    const unsigned long long kmask = (1ull << kKeyBits) - 1ull;
    for (;;) {
        if (tid == 0) sh.item = atomicAdd(counter, 1u);
        __syncthreads();
        const uint32_t it = sh.item;
        __syncthreads();
        if (it >= n) break;
        const uint32_t p = list[it];
        const PolyMeta M = meta[p];
        const CellWin W = window_of(M.mbr, g);
        const uint32_t T = M.T;
        const unsigned long long *sorted = sorted_all + M.key_off;
        unsigned long long *U = other_all + M.key_off;
        uint8_t *flags = flags_all + M.key_off;
        const uint32_t rows = (uint32_t)(W.wj1 - W.wj0 + 1);
        uint32_t *row_start = rb_all + M.rb_off;
        const unsigned long long *cross = cross_all + M.cross_off;
        if (tid == 0) mbr_out[p] = make_int4(M.mbr[0], M.mbr[1], M.mbr[2], M.mbr[3]);
        // 2. one key per cell (the last of a cell's run carries the crossed
        //    flag when any edge crossed it: (d << 1) | 1 sorts last)
        uint32_t carry = 0;
        for (uint32_t t0 = 0; t0 < T; t0 += kBB) {
            const uint32_t k = t0 + tid;
            bool last = false;
            unsigned long long key = 0;
            if (k < T) {
                key = sorted[k] & kmask;
                last = k + 1 == T || ((sorted[k + 1] & kmask) >> 1) != (key >> 1);
            }
            uint32_t total;
            const uint32_t pos = carry + block_scan(last ? 1u : 0u, total, sh);
            if (last) U[pos] = key;
            carry += total;
        }
        const uint32_t K = carry;

        // 3. row starts in the sorted crossings: row r's crossings are
        //    [row_start[r], row_start[r + 1]); every entry is written once, by
        //    the crossing that opens its row or the one that closes the list
        const uint32_t inc = M.inc;
        const unsigned long long rmask = (1ull << kCrossRowBits) - 1;
        if (inc == 0)
            for (uint32_t r = tid; r <= rows; r += kBB) row_start[r] = 0;
        for (uint32_t q = tid; q < inc; q += kBB) {
            const uint32_t r = (uint32_t)((cross[q] >> kCrossXBits) & rmask);
            const uint32_t rp = q ? (uint32_t)((cross[q - 1] >> kCrossXBits) & rmask) + 1u : 0u;
            for (uint32_t rr = rp; rr <= r; ++rr) row_start[rr] = q;
            if (q + 1 == inc)
                for (uint32_t rr = r + 1; rr <= rows; ++rr) row_start[rr] = inc;
        }
        __syncthreads();

        // 4. classification: bit 0 gap before the cell non-empty, bit 1 that
        //    gap Full, bit 2 the cell Full
        for (uint32_t u = tid; u < K; u += kBB) {
            const unsigned long long key = U[u];
            const uint64_t d = key >> 1;
            const uint64_t first_gap = u ? (U[u - 1] >> 1) + 1 : 0;
            uint8_t f = 0;
            uint32_t x, y;
            if (d > first_gap) {
                f |= 1;
                hilbert_cell(g.order, first_gap, x, y);
                if (inside_cell(x, y, M, W, g, row_start, cross)) f |= 2;
            }
            if (!(key & 1ull)) {
                hilbert_cell(g.order, d, x, y);
                if (inside_cell(x, y, M, W, g, row_start, cross)) f |= 4;
            }
            flags[u] = f;
        }
        if (tid == 0) {
            const uint64_t nxt = (U[K - 1] >> 1) + 1;
            bool tail = false;
            if (nxt < ncells) {
                uint32_t x, y;
                hilbert_cell(g.order, nxt, x, y);
                tail = inside_cell(x, y, M, W, g, row_start, cross);
            }
            sh.k_count = tail ? 1u : 0u;
        }
        __syncthreads();
        const bool tailF = sh.k_count != 0;

        // 5. intervals
        uint2 *Aout = iv_out + M.slot_off;
        uint2 *Fout = iv_out + M.slot_off + even_up((uint64_t)T + 1);
        uint32_t na = 0, nf = 0;
        {
            // A: a new interval at every cell after a non-empty gap that is not Full
            uint32_t ca = 0, cf = 0;
            for (uint32_t t0 = 0; t0 < K; t0 += kBB) {
                const uint32_t u = t0 + tid;
                const bool ok = u < K;
                const uint8_t f = ok ? flags[u] : 0;
                const uint64_t d = ok ? (U[u] >> 1) : 0;
                const uint64_t prev_end = (ok && u) ? (U[u - 1] >> 1) + 1 : 0;  // end of the previous cell
                const bool brk = ok && u > 0 && (f & 1) && !(f & 2);
                uint32_t ta;
                const uint32_t ia = ca + block_scan(brk ? 1u : 0u, ta, sh);
                if (brk) {
                    Aout[ia].y = (uint32_t)prev_end;  // the interval before closes
                    Aout[ia + 1].x = (uint32_t)d;
                }
                if (ok && u == 0) Aout[0].x = ((f & 1) && (f & 2)) ? 0u : (uint32_t)d;
                ca += ta;
                // F: slots gap(u) then cell(u); a run starts where an F slot
                // follows a non-F one and ends where a non-F one follows
                const bool gF = ok && (f & 2);
                const bool cF = ok && (f & 4);
                const bool prevCellF = ok && u > 0 && (flags[u - 1] & 4);
                const bool prev_of_cell = (f & 1) ? gF : prevCellF;
                bool next_of_cell = tailF;
                if (ok && u + 1 < K) {
                    const uint8_t fn = flags[u + 1];
                    next_of_cell = (fn & 1) ? (fn & 2) != 0 : (fn & 4) != 0;
                }
                const bool sg = gF && !prevCellF, sc = cF && !prev_of_cell;
                const bool eg = gF && !cF, ec = cF && !next_of_cell;
                uint32_t tf;
                const uint32_t i0 = cf + block_scan((sg ? 1u : 0u) + (sc ? 1u : 0u), tf, sh);
                if (sg) Fout[i0].x = (uint32_t)prev_end;                     // gap starts after the previous cell
                if (eg) Fout[i0 + (sg ? 1u : 0u) - 1u].y = (uint32_t)d;        // and ends at this cell
                if (sc) Fout[i0 + (sg ? 1u : 0u)].x = (uint32_t)d;
                if (ec) Fout[i0 + (sg ? 1u : 0u) + (sc ? 1u : 0u) - 1u].y = (uint32_t)(d + 1);
                cf += tf;
            }
            na = ca + 1;
            nf = cf;
            if (tid == 0) {
                const uint64_t last_end = (U[K - 1] >> 1) + 1;
                Aout[na - 1].y = (uint32_t)(tailF ? ncells : last_end);  // 2^32 wraps to 0 by design
                const bool lastCellF = (flags[K - 1] & 4) != 0;
                if (tailF) {
                    if (!lastCellF) Fout[nf].x = (uint32_t)last_end;
                    Fout[lastCellF ? nf - 1 : nf].y = (uint32_t)ncells;
                }
            }
            if (tailF && !(flags[K - 1] & 4)) nf += 1;
        }
        if (tid == 0) {
            uint32_t *dsc = desc_out + 4 * (size_t)p;
            dsc[0] = (uint32_t)M.slot_off;
            dsc[1] = na;
            dsc[2] = (uint32_t)(M.slot_off + even_up((uint64_t)T + 1));
            dsc[3] = nf;
        }
        __syncthreads();
    }
}

april_status cuda_fail(cudaError_t e, const char *what) {
    return fail(APRIL_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

inline uint64_t r256(uint64_t b) { return april_round256(b); }

// The work buffer: totals, 80 bytes per polygon (record and path lists), then
// what the sorted path would need for all polygons.  The polygons that take
// it use the front of each region; the tile records lie behind their keys (a
// tiled polygon has room for 8 bytes per touched cell there and needs 4).
constexpr uint64_t kPolyBytes = 80;
struct WorkLayout {
    uint64_t totals, meta, keys, tmp, flags, rb, cross, ctmp, hist, dbase, total;
};

inline uint32_t sort_tiles(uint64_t keys) { return (uint32_t)((keys + kRsTile - 1) / kRsTile); }

WorkLayout work_layout(uint32_t n, uint64_t keys, uint64_t rb, uint64_t cross) {
    WorkLayout L{};
    uint64_t o = 0;
    L.totals = o;
    o += 256;
    L.meta = o;
    o += r256((uint64_t)n * kPolyBytes);
    const uint64_t min_total = o;
    L.keys = o;
    o += r256(keys * 8);
    L.tmp = o;
    o += r256(keys * 8);
    L.flags = o;
    o += r256(keys);
    L.rb = o;
    o += r256(rb * 4);
    L.cross = o;
    o += r256(cross * 8);
    L.ctmp = o;
    o += r256(cross * 8);
    L.hist = o;
    o += r256((uint64_t)256 * sort_tiles(std::max(keys, cross)) * 4);
    L.dbase = o;
    o += 1024;
    L.total = keys || rb ? o : min_total;
    return L;
}

}  // namespace

// The sorted path for the h.count[kSorted] polygons of `list`.
static cudaError_t build_sorted(char *work, const WorkLayout &L, const uint32_t *list, const Totals &h, uint32_t n_polys,
                                const int2 *xy, const uint64_t *off, const GridP &g, const PolyMeta *meta, Totals *tot,
                                uint32_t *desc, int4 *mbr, uint2 *iv, uint64_t sms, cudaStream_t s) {
    const uint32_t n = h.count[kSorted];
    int occ = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_bconstruct, kBB, 0);
    const unsigned grid = (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(n, sms * (uint64_t)std::max(occ, 1)));
    auto *keys = (unsigned long long *)(work + L.keys), *tmp = (unsigned long long *)(work + L.tmp);
    k_bemit<<<grid, kBB, 0, s>>>(xy, off, list, n, g, meta, keys, (unsigned long long *)(work + L.cross),
                                 &tot->ctr_emit);
    cudaError_t e = cudaGetLastError();
    // one radix sort of all cell keys (the polygon id sits above the 33 key
    // bits) and one of all crossing keys (above row and x)
    uint32_t pbits = 0;
    while (pbits < 32 && (1ull << pbits) < n_polys) ++pbits;
    auto *hist = (uint32_t *)(work + L.hist), *dbase = (uint32_t *)(work + L.dbase);
    auto radix_sort = [&](unsigned long long *a, unsigned long long *t, uint64_t N, uint32_t bits) {
        const uint32_t passes = (bits + 7) / 8, ntiles = sort_tiles(N);
        const unsigned gs = (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(ntiles, sms * 8));
        for (uint32_t pass = 0; pass < passes && N && e == cudaSuccess; ++pass) {
            k_rs_hist<<<gs, kRsT, 0, s>>>(a, N, 8 * pass, hist, ntiles);
            k_rs_rows<<<256, kRsScanT, 0, s>>>(hist, ntiles, dbase);
            k_rs_digits<<<1, 256, 0, s>>>(dbase);
            k_rs_scatter<<<gs, kRsT, 0, s>>>(a, t, N, 8 * pass, hist, dbase, ntiles);
            e = cudaGetLastError();
            std::swap(a, t);
        }
        return a;  // the buffer holding the sorted keys
    };
    unsigned long long *src = radix_sort(keys, tmp, h.skeys, kKeyBits + pbits);
    unsigned long long *dst = src == keys ? tmp : keys;
    const unsigned long long *csorted = radix_sort((unsigned long long *)(work + L.cross),
                                                   (unsigned long long *)(work + L.ctmp), h.scross,
                                                   kCrossPolyShift + pbits);
    if (e == cudaSuccess) {
        k_bconstruct<<<grid, kBB, 0, s>>>(xy, off, list, n, g, meta, src, dst, csorted, (uint8_t *)(work + L.flags),
                                          (uint32_t *)(work + L.rb), desc, mbr, iv, &tot->ctr_build);
        e = cudaGetLastError();
    }
    return e;
}

int april_build_wait_limit(uint32_t spins) {
    const uint32_t v = std::min(spins, kTileSpins);
    return (int)cudaMemcpyToSymbol(c_tile_spins, &v, sizeof v);
}

extern "C" april_status april_build_sets_device(april_ctx *ctx, const int32_t *d_xy, const uint64_t *d_vert_off,
                                                uint32_t n_polys, const april_grid *grid, void *d_work,
                                                size_t work_bytes, void *d_image, size_t image_bytes,
                                                april_dev_sets *out, april_device_build_info *info, void *stream) {
    if (!ctx || !info || !out) return fail(APRIL_ERR_INVALID_ARG, "NULL argument");
    *info = april_device_build_info{};
    GridP g{};
    april_status st = april::check_grid_params(grid, g.ox, g.oy, g.h, g.order, g.G);
    if (st) return st;
    if (n_polys == 0) return fail(APRIL_ERR_INVALID_ARG, "no polygons");
    if (!d_xy || !d_vert_off) return fail(APRIL_ERR_INVALID_ARG, "NULL polygon arrays");
    if ((((uintptr_t)d_xy) & 7u) || (((uintptr_t)d_vert_off) & 7u))
        return fail(APRIL_ERR_INVALID_ARG, "polygon arrays must be 8-byte aligned");
    const WorkLayout L0 = work_layout(n_polys, 0, 0, 0);
    info->work_bytes = L0.total;
    if (!d_work || work_bytes < L0.total) return fail(APRIL_ERR_OVER_BUDGET, "work buffer below the counting size");
    if (((uintptr_t)d_work) & 255u) return fail(APRIL_ERR_INVALID_ARG, "work buffer must be 256-byte aligned");
    cudaStream_t s = (cudaStream_t)stream;
    char *work = (char *)d_work;
    auto *tot = (Totals *)(work + L0.totals);
    auto *meta = (PolyMeta *)(work + L0.meta);
    auto *lists = (uint32_t *)(work + L0.meta + (uint64_t)n_polys * sizeof(PolyMeta));  // kPaths lists of n_polys
    cudaError_t e = cudaMemsetAsync(tot, 0, sizeof(Totals), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(&tot->first_err, 0xFF, 8, s);
    const uint64_t sms = (uint64_t)april_ctx_num_sms(ctx);
    const int l2h = (int)grid->log2_cell;
    auto resident = [&](const void *kernel, uint64_t want) {  // CTAs: what is resident at once, no more than wanted
        int occ = 1;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, kBB, 0);
        return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(want, sms * (uint64_t)std::max(occ, 1)));
    };
    if (e == cudaSuccess) {
        const uint32_t nb = (n_polys + kPlace - 1) / kPlace;
        // with enough polygons to fill the chip several times over, only the
        // largest are worth cutting up; with few, one warp's polygon would be the last
        const uint64_t big_verts = n_polys >= 64 * sms ? 1024 : 64;
        k_bcount<<<resident((const void *)k_bcount, ((uint64_t)n_polys + kBW - 1) / kBW), kBB, 0, s>>>(
            (const int2 *)d_xy, d_vert_off, n_polys, g, l2h, meta, tot, lists, big_verts);
        k_bcount_big<<<resident((const void *)k_bcount_big, ~0ull), kBB, 0, s>>>((const int2 *)d_xy, d_vert_off, g, l2h,
                                                                               meta, tot, lists);
        k_bcount_end<<<resident((const void *)k_bcount_end, ((uint64_t)n_polys + kBW - 1) / kBW), kBB, 0, s>>>(
            (const int2 *)d_xy, d_vert_off, g, meta, tot, lists);
        k_bsum<<<nb, 256, 0, s>>>(d_vert_off, meta, n_polys, g, tot);
        k_btop<<<1, 1024, 0, s>>>(meta, nb, tot);
        k_bplace<<<nb, 256, 0, s>>>(d_vert_off, meta, n_polys, g, tot, lists);
        e = cudaGetLastError();
    }
    Totals h{};
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, tot, sizeof h, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e, "counting cells on the device");
    if (h.n_err) {
        char m[160];
        const uint32_t code = (uint32_t)(h.first_err & 0xFF), first = (uint32_t)(h.first_err >> 8);
        const char *why = code == 1   ? "fewer than 3 vertices (or offsets not monotone)"
                          : code == 2 ? "outside the grid"
                          : code == 4 ? "meets no cell"
                                      : "too large (2^31 cells, or an MBR 2^26 lattice units wide)";
        std::snprintf(m, sizeof m, "polygon %u: %s (%u polygons rejected)", first, why, h.n_err);
        return fail(code == 3 ? APRIL_ERR_INVALID_ARG : APRIL_ERR_GEOMETRY, m);
    }
    const WorkLayout L = work_layout(n_polys, h.keys, h.rb, h.cross);
    const uint64_t desc_b = r256((uint64_t)n_polys * 16), mbr_b = r256((uint64_t)n_polys * 16);
    const uint64_t iv_b = r256(h.slots * 8 + 16), posts_b = r256(april_posts_words(h.slots) * 4);
    const uint64_t img = desc_b + mbr_b + iv_b + posts_b;
    info->touched_cells = h.keys;
    info->work_bytes = L.total;
    info->image_bytes = img;
    info->iv_slots = h.slots;
    if (h.slots > 0xFFFFFFF0ull) return fail(APRIL_ERR_INVALID_ARG, "more than 2^32 interval slots in one set");
    if (h.keys > 0xFFFFFFFFull || h.cross > 0xFFFFFFFFull || n_polys > (1u << 22))
        return fail(APRIL_ERR_INVALID_ARG, "more than 2^32 - 1 cells or crossings, or 2^22 polygons, in one build");
    if (work_bytes < L.total) return fail(APRIL_ERR_OVER_BUDGET, "work buffer too small");
    if (!d_image || image_bytes < img) return fail(APRIL_ERR_OVER_BUDGET, "image buffer too small");
    if (((uintptr_t)d_image) & 255u) return fail(APRIL_ERR_INVALID_ARG, "image buffer must be 256-byte aligned");
    char *image = (char *)d_image;
    const int2 *xy = (const int2 *)d_xy;
    auto *desc = (uint32_t *)image;
    auto *mbr = (int4 *)(image + desc_b);
    auto *iv = (uint2 *)(image + desc_b + mbr_b);
    const uint32_t n_tiled = (uint32_t)(h.tiled >> 40), records = (uint32_t)(h.tiled & ((1ull << 40) - 1));
    if (n_tiled) {
        auto *recs = (TileRec *)(work + L.keys + r256(h.skeys * 8));
        const uint32_t *list = lists + (uint64_t)kTiled * n_polys;
        k_btinit<<<resident((const void *)k_btinit, (n_tiled + kBW - 1) / kBW), kBB, 0, s>>>(list, n_tiled, g, meta, recs);
        k_btile<<<resident((const void *)k_btile, records), kBB, 0, s>>>(xy, d_vert_off, records, g, l2h, meta, recs,
                                                                         &tot->ctr_tile, april_ctx_status_word(ctx), desc,
                                                                         mbr, iv);
    }
    if (h.count[kMid])
        k_bmid<<<resident((const void *)k_bmid, h.count[kMid]), kBB, 0, s>>>(
            xy, d_vert_off, lists + (uint64_t)kMid * n_polys, h.count[kMid], g, l2h, meta, desc, mbr, iv);
    if (h.count[kSmall])
        k_bsmall<<<resident((const void *)k_bsmall, (h.count[kSmall] + kBW - 1) / kBW), kBB, 0, s>>>(
            xy, d_vert_off, lists + (uint64_t)kSmall * n_polys, h.count[kSmall], g, l2h, meta, desc, mbr, iv);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess && h.count[kSorted])
        e = build_sorted(work, L, lists + (uint64_t)kSorted * n_polys, h, n_polys, xy, d_vert_off, g, meta, tot, desc,
                         mbr, iv, sms, s);
    if (e == cudaSuccess)  // the skip index of the interval array
        e = (cudaError_t)april_launch_posts((const uint32_t *)(image + desc_b + mbr_b), h.slots,
                                            (uint32_t *)(image + desc_b + mbr_b + iv_b), s);
    if (e != cudaSuccess) return cuda_fail(e, "building lists on the device");
    *out = april_dev_sets{};
    out->desc = (const uint32_t *)image;
    out->iv = (const uint32_t *)(image + desc_b + mbr_b);
    out->mbr = (const int32_t *)(image + desc_b);
    out->posts = (const uint32_t *)(image + desc_b + mbr_b + iv_b);
    out->n_objects = n_polys;
    out->order = g.order;
    out->iv_slots = h.slots;
    out->n_entries = n_polys;
    out->grid_ox = g.ox;
    out->grid_oy = g.oy;
    out->grid_log2_cell = grid->log2_cell;
    out->grid_known = 1;
    out->grid_id = april_grid_id(g.ox, g.oy, grid->log2_cell, g.order);
    return APRIL_OK;
}
