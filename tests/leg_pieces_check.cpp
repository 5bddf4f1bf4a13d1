// leg_pieces against the search over every count.
#include <cstdio>

#include "batch_tiles.h"

using namespace gmg::batch;

static int every_count(int64_t columns, int64_t slots, int len, int unit, int extra) {
    int best = 1;
    int64_t cost = INT64_MAX;
    for (int p = 1; p <= len; ++p) {
        const int64_t waves = (columns * p + slots - 1) / slots;
        const int64_t c = waves * ((int64_t)unit * ((len + p - 1) / p) + extra);
        if (c < cost) {
            best = p;
            cost = c;
        }
    }
    return best;
}

int main() {
    long long checked = 0;
    for (int len : {1, 2, 3, 5, 7, 15, 31, 32, 63, 100, 127, 255, 511, 1023, 8191})
        for (int64_t slots : {1, 152, 304, 1216, 24320})
            for (int64_t columns : {1, 2, 3, 7, 50, 285, 1000, 5000, 100000})
                for (int unit = 1; unit <= 2; ++unit) {
                    const int a = leg_pieces(columns, slots, len, unit, 2 * unit),
                              e = every_count(columns, slots, len, unit, 2 * unit);
                    ++checked;
                    if (a != e) {
                        std::printf("len %d slots %lld columns %lld: %d, every count %d\n", len,
                                    (long long)slots, (long long)columns, a, e);
                        return 1;
                    }
                }
    std::printf("checked %lld\n", checked);
    return 0;
}
