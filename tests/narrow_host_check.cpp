// cvt::narrow against the C cast, bit for bit: random significands over every
// exponent the float format rounds, underflows and overflows at, ties to even
// and their neighbours, both signs, zeros, infinities.  Prints the mismatches.
#include <cmath>
#include <cstdio>
#include <limits>
#include <random>

#include "df.cuh"

static long long bad = 0, checked = 0;
static void check(double x) {
    const float a = gmg::cvt::narrow(x), b = (float)x;
    ++checked;
    if (gmg::cvt::f_bits(a) != gmg::cvt::f_bits(b) && !(std::isnan(a) && std::isnan(b)))
        if (bad++ < 10) std::printf("%a: %a, cast %a\n", x, a, b);
}

int main() {
    std::mt19937_64 g(7);
    for (int e = 1023 - 160; e <= 1023 + 135; ++e)
        for (int k = 0; k < 20000; ++k) {
            const uint64_t frac = g() >> 12;
            const uint64_t top = frac & ~0x1fffffffull;
            const uint64_t fs[8] = {frac, top, top | 0x10000000u, top | 0x0fffffffu, top | 0x10000001u,
                                    0xfffffffffffffu, 0xffffff0000000u, 0xfffffefffffffu};
            for (uint64_t f : fs)
                for (int s = 0; s < 2; ++s)
                    check(gmg::cvt::bits_d((uint64_t)s << 63 | (uint64_t)e << 52 | f));
        }
    for (double x : {0.0, -0.0, std::numeric_limits<double>::infinity(),
                     -std::numeric_limits<double>::infinity(), std::numeric_limits<double>::quiet_NaN(),
                     std::numeric_limits<double>::denorm_min(), std::numeric_limits<double>::max()})
        check(x);
    std::printf("checked %lld, mismatches %lld\n", checked, bad);
    return bad != 0;
}
