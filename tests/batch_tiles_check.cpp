// Cutting of a level into the batched legs' tiles: every coarse node and every
// fine row is written by exactly one tile, a tile holds all rows that its
// outputs depend on, and no piece of the marching direction is empty.
#include <cstdio>

#include "batch_tiles.h"

using namespace gmg::batch;

static int fail(const char* what, int n, int R) {
    std::printf("%s n=%d R=%d\n", what, n, R);
    return 1;
}

int main() {
    for (int n = 4; n <= 16384; n *= 2) {
        const int nc = n / 2, G = n / 4;
        for (int down = 0; down < 2; ++down) {
            const int th = leg_threads(n, down), R = leg_rows(n, th);
            if (th % 32 || th > 640 || th % std::min(G, 32)) return fail("threads", n, th);
            if (n <= 64 && R < n) return fail("one tile", n, R);
        }
        for (int R : {12, 16, 32, 34, 38, 40, 64, 128}) {
            std::vector<int> fine(n + 1), coarse(nc + 1), up(n + 1);
            for (const Rows& t : rows_down(n, R)) {
                if (t.y0 % 2 || t.y0 < 0 || t.jb <= t.ja) return fail("down tile", n, R);
                const bool lo = t.y0 == 0, hi = t.y0 + R >= n;
                for (int J = t.ja; J < t.jb; ++J) {
                    ++coarse[J];
                    // u0 of 2J - 3 .. 2J + 3, or as far as the boundary
                    if (!lo && 2 * J - 3 < t.y0) return fail("down below", n, R);
                    if (!hi && 2 * J + 3 > t.y0 + R - 1) return fail("down above", n, R);
                }
                for (int y = 2 * t.ja - 1; y <= 2 * t.jb - 2 + (t.jb == nc); ++y) {
                    ++fine[y];
                    if ((!lo && y - 1 < t.y0) || (!hi && y + 1 > t.y0 + R - 1))
                        return fail("down sweep", n, R);
                }
            }
            for (const Rows& t : rows_up(n, R)) {
                if (t.y0 % 2 || t.y0 < 0 || t.jb <= t.ja) return fail("up tile", n, R);
                for (int y = t.ja; y < t.jb; ++y) {
                    ++up[y];
                    if (y - 1 < t.y0 || (y + 1 > t.y0 + R - 1 && y + 1 < n))
                        return fail("up rows", n, R);
                }
            }
            for (int y = 1; y < n; ++y)
                if (fine[y] != 1 || up[y] != 1) return fail("fine rows", n, R);
            for (int J = 1; J < nc; ++J)
                if (coarse[J] != 1) return fail("coarse rows", n, R);
        }
        std::vector<int> groups(G);
        for (int g0 : leg_columns(G, 30))
            for (int l = 0; l < 32; ++l) {
                const int g = g0 + l;
                if (g >= 0 && g < G && (G <= 32 || (l >= 1 && l <= 30))) ++groups[g];
            }
        for (int g = 0; g < G; ++g)
            if (groups[g] != 1) return fail("groups", n, g);
        for (int64_t columns : {1, 7, 285, 5000})
            for (int len : {nc - 1, n - 1}) {
                const int p = leg_pieces(columns, 304, len, 2, 4);
                if (p < 1 || p > len) return fail("pieces", n, p);
            }
    }
    std::printf("ok\n");
    return 0;
}
