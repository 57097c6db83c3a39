// Rasterising an edge row by row for the GPU builder (build_device.cu): the
// cells of every grid row it touches and enters, and where it crosses the
// row's centre line, in 32-bit coordinates relative to the grid's origin.
// The results are geom.h's (edge_cells_in_row, enters_open_square,
// centre_rows) for coordinates below 2^28 in magnitude and cells of at most
// 2^24 lattice units.
#pragma once
#include <cstdint>

#include "geom.h"

namespace april_geom {

// An edge oriented upwards, relative to the grid's origin.
struct EdgeRel {
    int32_t ax, ay, bx, by;
};

APRIL_HD EdgeRel edge_rel(int32_t ax, int32_t ay, int32_t bx, int32_t by) {
    if (ay > by || (ay == by && ax > bx)) return EdgeRel{bx, by, ax, ay};
    return EdgeRel{ax, ay, bx, by};
}

// num = q den + r with 0 <= r < den, for |num / den| at most 2^26: a quotient
// estimated in float (inv ~ 1 / den, each factor within 2^-24) is at most 17
// off, the estimate of its remainder's quotient one, and the remainder itself
// says which.  Larger quotients would not end: the estimates saturate and the
// last loops step down by ones.
APRIL_HD void floor_divmod(int64_t num, int32_t den, float inv, int32_t &q, int32_t &r) {
    const int32_t q0 = (int32_t)((float)num * inv);
    int64_t rem = num - (int64_t)q0 * den;
    int32_t q1 = (int32_t)((float)rem * inv);
    rem -= (int64_t)q1 * den;
    while (rem < 0) rem += den, --q1;
    while (rem >= den) rem -= den, ++q1;
    q = q0 + q1;
    r = (int32_t)rem;
}

// The same for |num| below 2^31, in 32 bits: the estimate is at most one off
// for |num / den| below 2^22, at most 17 up to 2^26.
APRIL_HD void floor_divmod32(int32_t num, int32_t den, float inv, int32_t &q, int32_t &r) {
    q = (int32_t)((float)num * inv);
    r = num - q * den;
    while (r < 0) r += den, --q;
    while (r >= den) r -= den, ++q;
}

// Rows [j0, j1] of the grid (cells of 2^l, G rows) whose closed strip the
// edge meets.
APRIL_HD void rel_rows(const EdgeRel &e, int l, int32_t G, int32_t &j0, int32_t &j1) {
    const int32_t h1 = (1 << l) - 1;
    j0 = ((e.ay + h1) >> l) - 1;
    j1 = e.by >> l;
    if (j0 < 0) j0 = 0;
    if (j1 > G - 1) j1 = G - 1;
}

// Rows [r0, r1] whose centre line the edge crosses (lower end included, upper not).
APRIL_HD void rel_centre_rows(const EdgeRel &e, int l, int32_t &r0, int32_t &r1) {
    const int32_t up = (1 << l) - 1 - (1 << (l - 1));
    r0 = (e.ay + up) >> l;
    r1 = ((e.by + up) >> l) - 1;
}

// What an edge does in one row: it touches the closed cells [i0, i1], enters
// the open squares of [c0, c1], and, where `turns`, crosses the centre line at
// an x that lies left of the centres of exactly the cells from `t` on.  The
// columns are not clipped to the grid.
struct RowCells {
    int32_t j, i0, i1, c0, c1, t;
    bool turns;
};

// Calls f(RowCells) for the rows [ja, jb] (within rel_rows) in order, of an
// edge at most 2^26 wide.  The edge's x on a row line is kept as quotient and
// remainder over its height and stepped by half rows, so a run of rows takes
// two divisions.  Every height divided is at most the edge's own, so the
// quotients stay within its width: an edge no higher than half a row spans no
// two half-row lines, and its step, which no row would use, is left out.
template <class F>
APRIL_HD void edge_walk(const EdgeRel &e, int l, int32_t ja, int32_t jb, F f) {
    const int32_t h = 1 << l, hh = h >> 1, h1 = h - 1;
    const int32_t den = e.by - e.ay, dx = e.bx - e.ax;
    if (den == 0) {
        for (int32_t j = ja; j <= jb; ++j) {
            const int32_t y0 = j << l;
            const bool in = y0 < e.ay && e.ay < y0 + h && e.ax < e.bx;  // a point enters nothing (geom.h)
            f(RowCells{j, ((e.ax + h1) >> l) - 1, e.bx >> l, in ? e.ax >> l : 1, in ? ((e.bx + h1) >> l) - 1 : 0, 0,
                       false});
        }
        return;
    }
    const float inv = 1.0f / (float)den;
    // x at a height y above ay is ax + y dx / den; most edges' products fit 32 bits
    const int64_t big = (int64_t)den * (dx < 0 ? -(int64_t)dx : dx);
    const bool fits = big < (1ll << 31);
    auto at = [&](int32_t y, int32_t &qq, int32_t &rr) {
        if (fits) floor_divmod32(y * dx, den, inv, qq, rr);
        else floor_divmod((int64_t)y * dx, den, inv, qq, rr);
    };
    int32_t hq = 0, hr = 0;  // the step of half a row
    if (den > hh) at(hh, hq, hr);
    int32_t y0 = ja << l, q = e.ax, r = 0;  // x at max(y0, ay) = q + r / den
    bool line = y0 > e.ay;                  // that is the row's lower line
    if (line) {
        at(y0 - e.ay, q, r);
        q += e.ax;
    }
    for (int32_t j = ja; j <= jb; ++j) {
        const int32_t y1 = y0 + h, yc = y0 + hh;
        int32_t q1 = e.bx, r1 = 0, qc = q, rc = r;
        if (line) {
            qc += hq;
            rc += hr;
            if (rc >= den) rc -= den, ++qc;
        }
        if (y1 < e.by) {
            if (line) {
                q1 = qc + hq;
                r1 = rc + hr;
                if (r1 >= den) r1 -= den, ++q1;
            } else {
                at(y1 - e.ay, q1, r1);
                q1 += e.ax;
            }
        }
        const bool turns = e.ay <= yc && yc < e.by;
        if (turns && !line) {
            if (y1 < e.by) {
                qc = q1 - hq;
                rc = r1 - hr;
                if (rc < 0) --qc;
            } else {
                at(yc - e.ay, qc, rc);
                qc += e.ax;
            }
        }
        const int32_t ql = dx >= 0 ? q : q1, rl = dx >= 0 ? r : r1, qh = dx >= 0 ? q1 : q, rh = dx >= 0 ? r1 : r;
        const bool lon = rl == 0 && !(ql & h1), hon = rh == 0 && !(qh & h1);  // on a column line
        const bool in = (e.ay > y0 ? e.ay : y0) < (e.by < y1 ? e.by : y1);
        f(RowCells{j, (ql >> l) - (lon ? 1 : 0), qh >> l, in ? ql >> l : 1, in ? (qh >> l) - (hon ? 1 : 0) : 0,
                   (qc + hh) >> l, turns});
        q = q1;
        r = r1;
        y0 = y1;
        line = true;
    }
}

// The state of the Hilbert walk (geom.h's symmetries) and the id of square
// (x, y) after `levels` levels from the top.
APRIL_HD uint32_t hilbert_id_state(uint32_t levels, uint32_t x, uint32_t y, uint32_t &s) {
    uint32_t d = 0;
    s = 0;
    for (int k = (int)levels - 1; k >= 0; --k) {
        uint32_t bx = (x >> k) & 1u, by = (y >> k) & 1u;
        apply_sym(s, bx, by);
        const uint32_t digit = (bx << 1) | (bx ^ by);
        d = (d << 2) | digit;
        s ^= digit == 0 ? 1u : digit == 3 ? 2u : 0u;
    }
    return d;
}

// Square number d, of 4^levels, of a walk that starts in state s: its place
// and the state inside it.
APRIL_HD void hilbert_square(uint32_t levels, uint32_t d, uint32_t &s, uint32_t &x, uint32_t &y) {
    x = y = 0;
    for (int k = (int)levels - 1; k >= 0; --k) {
        const uint32_t digit = (d >> (2 * k)) & 3u;
        uint32_t bx = digit >> 1, by = (digit >> 1) ^ (digit & 1u);
        apply_sym(s, bx, by);
        x = 2 * x + bx;
        y = 2 * y + by;
        s ^= digit == 0 ? 1u : digit == 3 ? 2u : 0u;
    }
}

// Table for a 4 x 4 block's Hilbert order: entry [state][half][cells] is the
// 16-bit set of the walk's positions of the cells in rows 2 half (low nibble)
// and 2 half + 1 (high nibble).
APRIL_HD uint16_t hilbert_rows(uint32_t s, uint32_t half, uint32_t cells) {
    uint32_t m = 0;
    for (uint32_t d = 0; d < 16; ++d) {
        uint32_t t = s, x, y;
        hilbert_square(2, d, t, x, y);
        if (y >> 1 == half && ((cells >> (4 * (y & 1u) + x)) & 1u)) m |= 1u << d;
    }
    return (uint16_t)m;
}

// The 64 cells of an 8 x 8 block (lo: rows 0 to 3, hi: 4 to 7, a byte each) in
// the order of a walk that starts in state s; tab is hilbert_rows' table.
template <class Tab>
APRIL_HD uint64_t block_in_order(const Tab &tab, uint32_t s, uint32_t lo, uint32_t hi) {
    uint32_t w[4];
    for (uint32_t d = 0; d < 4; ++d) {
        uint32_t bx = d >> 1, by = (d >> 1) ^ (d & 1u);
        apply_sym(s, bx, by);
        const uint32_t t = s ^ (d == 0 ? 1u : d == 3 ? 2u : 0u);
        const uint32_t v = ((by ? hi : lo) >> (4 * bx)) & 0x0F0F0F0Fu, c = v | v >> 4;
        w[d] = tab(t, 0, c & 0xFFu) | tab(t, 1, (c >> 16) & 0xFFu);
    }
    return (uint64_t)(w[0] | w[1] << 16) | (uint64_t)(w[2] | w[3] << 16) << 32;
}

}  // namespace april_geom
