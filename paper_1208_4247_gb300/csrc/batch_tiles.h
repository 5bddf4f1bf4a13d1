// How the batched legs cut a level of n^d cells into tiles: rows of y for the
// 3D kernels' CTAs, pieces of the marching direction for all.  Plain C++.
#pragma once

#include <algorithm>
#include <cstdint>
#include <vector>

namespace gmg {
namespace batch {

struct Rows {
    int y0;      // first row held; even
    int ja, jb;  // down: coarse rows [ja, jb); up: fine rows [ja, jb)
};

// A tile holds R rows (even).  Down: r of row y needs u1 of y - 1 .. y + 1 and
// so u0 of y - 2 .. y + 2, a coarse row J needs r of 2J - 1 .. 2J + 1; at row 0
// and row n nothing beyond is needed.  Up: row y needs y - 1 .. y + 1.
inline std::vector<Rows> rows_down(int n, int R) {
    std::vector<Rows> v;
    const int nc = n / 2;
    for (int ja = 1; ja < nc;) {
        const int y0 = std::max(0, 2 * ja - 4);
        const int jb = y0 + R >= n ? nc : (y0 + R - 4) / 2 + 1;
        v.push_back({y0, ja, jb});
        ja = jb;
    }
    return v;
}
inline std::vector<Rows> rows_up(int n, int R) {
    std::vector<Rows> v;
    for (int ja = 1; ja < n;) {
        const int y0 = ja - 1;
        const int jb = y0 + R >= n ? n : y0 + R - 1;
        v.push_back({y0, ja, jb});
        ja = jb;
    }
    return v;
}

// What the 3D legs are compiled for (launch bounds, shared memory).
constexpr int kLegThreads = 512;

// Threads of a 3D leg's CTA: n / 4 lanes per row (at most 32) times the pairs
// of rows.  Levels up to n = 64 are one tile; above, the number of warps (one
// pair of rows each) that holds the fewest rows in all, the halo rows of the
// tiles counted, of up to 16 warps: with more, the registers of a thread (16384 a
// scheduler) hold a plane's loads for one step only.
inline int leg_threads(int n, bool down) {
    if (n <= 16) return 32;
    if (n <= 32) return 128;
    if (n <= 64) return kLegThreads;
    int best = 0;
    int64_t cost = 0;
    for (int w = kLegThreads / 32; w >= 12; --w) {
        const int64_t c = (int64_t)2 * w * (down ? rows_down(n, 2 * w) : rows_up(n, 2 * w)).size();
        if (!best || c < cost) {
            best = w;
            cost = c;
        }
    }
    return 32 * best;
}
inline int leg_rows(int n, int threads) { return 2 * (threads / std::min(n / 4, 32)); }

// Pieces of a marching direction of len steps for `columns` independent walks,
// `slots` of which run at once, each piece costing extra steps more: the count
// that makes the waves times the steps of one least.
inline int leg_pieces(int64_t columns, int64_t slots, int len, int unit, int extra) {
    int best = 1;
    int64_t cost = INT64_MAX;
    // of the counts that give pieces of seg steps only the least can win
    for (int p = 1; p <= len;) {
        const int seg = (len + p - 1) / p;
        const int64_t waves = (columns * p + slots - 1) / slots;
        const int64_t c = waves * ((int64_t)unit * seg + extra);
        if (c < cost) {
            best = p;
            cost = c;
        }
        if (seg == 1) break;
        p = (len + seg - 2) / (seg - 1);
    }
    return best;
}

// groups of the first lane in a row of G groups: one piece up to 32, beyond
// that `core` groups a piece behind a halo group
inline std::vector<int> leg_columns(int G, int core) {
    std::vector<int> v;
    if (G <= 32)
        v.push_back(0);
    else
        for (int g = 0; g < G; g += core) v.push_back(g - 1);
    return v;
}

}  // namespace batch
}  // namespace gmg
