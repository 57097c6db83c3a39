// raster.h's row walk against geom.h's exact predicates, on the host: for
// every grid order, edges of small and large heights and slopes in both
// directions, at and between the grid's lines.  Prints the rows compared.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "../paper_2307_01716_gb300/csrc/raster.h"

using namespace april_geom;

static void die(const char *what, const EdgeRel &e, int l, const RowCells &c) {
    std::printf("%s: edge (%d, %d) (%d, %d), cells of 2^%d, row %d: touches [%d, %d], enters [%d, %d], turns %d at %d\n",
                what, e.ax, e.ay, e.bx, e.by, l, c.j, c.i0, c.i1, c.c0, c.c1, (int)c.turns, c.t);
    std::exit(1);
}

int main() {
    std::mt19937_64 g(7);
    long rows = 0;
    for (int order = 1; order <= 16; ++order)
        for (int l : {24 - order, 26 - order}) {
            if (l > 24 || l < 1) continue;
            const int32_t h = 1 << l, hh = h / 2, G = 1 << order;
            std::vector<int64_t> dens{0, 1, 2, 3, 100, hh - 1, hh, hh + 1, h - 1, h, h + 1, 2 * h + 1, 5 * h + 3};
            std::vector<int64_t> dxs{0, 1, h - 1, h, h + 1, 1 << 20, 1 << 22, (1 << 26) - 1, (int64_t)(g() >> 39)};
            for (int64_t den : dens)
                for (int64_t dx : dxs)
                    for (int rep = 0; rep < 24; ++rep) {
                        // the lower end near a row line, a centre line or anywhere; both slopes
                        const int64_t row = (int64_t)(g() % (uint64_t)G), at = row * h;
                        const int64_t off[] = {0, 1, -1, hh, hh - 1, (int64_t)(g() % (uint64_t)h), -(den / 2), h - den};
                        const int64_t ay = at + off[rep % 8], by = ay + den;
                        const int64_t xoff[] = {0, 1, hh, (int64_t)(g() % (uint64_t)h)};
                        int64_t ax = (int64_t)(g() % (uint64_t)G) * h + xoff[g() % 4], bx = ax + (rep & 1 ? -dx : dx);
                        if (std::max(std::llabs(ax), std::llabs(bx)) >= 1 << 28 || by >= 1 << 28) continue;
                        const EdgeRel e = edge_rel((int32_t)ax, (int32_t)ay, (int32_t)bx, (int32_t)by);
                        const EdgeUp u = edge_up(ax, ay, bx, by);
                        int32_t j0, j1;
                        rel_rows(e, l, G, j0, j1);
                        if (j1 < j0) continue;
                        const int32_t ja = j0 + (int32_t)(g() % (uint64_t)(j1 - j0 + 1));
                        edge_walk(e, l, ja, std::min(j1, ja + 7), [&](const RowCells &c) {
                            ++rows;
                            // geom.h clips to a grid: shift the columns into one that holds all of them
                            const int64_t sh = (1ll << 29) >> l << l, ncol = 1ll << (30 - l);
                            const EdgeUp w{u.ax + sh, u.ay, u.bx + sh, u.by};
                            int64_t i0, i1, r0, r1;
                            const bool any = edge_cells_in_row(w, 0, 0, h, ncol, c.j, i0, i1);
                            if (any ? i0 - sh / h != c.i0 || i1 - sh / h != c.i1 : c.i0 <= c.i1) die("touched", e, l, c);
                            for (int64_t i = (int64_t)c.i0 - 1; i <= (int64_t)c.i1 + 1; ++i) {
                                if (i > c.i0 + 3 && i < (int64_t)c.i1 - 3) i = (int64_t)c.i1 - 3;
                                const bool in = enters_open_square(u.ax, u.ay, u.bx, u.by, i * h, (int64_t)c.j * h, h);
                                if (in != (i >= c.c0 && i <= c.c1)) die("entered", e, l, c);
                            }
                            centre_rows(u, 0, h, -(1ll << 40), 1ll << 40, r0, r1);
                            if (c.turns != (c.j >= r0 && c.j <= r1)) die("turns", e, l, c);
                            if (c.turns) {
                                const int64_t yc = (int64_t)c.j * h + hh, dn = u.by - u.ay;
                                const int64_t x = floor_div(u.ax * dn + (yc - u.ay) * (u.bx - u.ax), dn);
                                const int64_t t = c.t;
                                if (t * h + hh <= x || (t - 1) * h + hh > x) die("turned at", e, l, c);
                            }
                        });
                    }
        }
    std::printf("%ld rows\n", rows);
    return 0;
}
