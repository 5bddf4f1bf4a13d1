// narrow_sixth(x) against x / 6 in long double: every exponent of the quotient a
// float rounds, underflows and overflows at, both signs, zeros, infinities, NaN.
//
// Bound in ulps: half of one and the 2^-47 before it (2^-22 ulp; and as much for
// the reference).  Subnormal quotients are rounded to 24 bits first: half of
// 2^-149 and at most a quarter of it before.
#include <cmath>
#include <cstdio>
#include <limits>
#include <random>

#include "df.cuh"

static long long bad = 0, checked = 0;
static void fail(double x, float got) {
    if (bad++ < 10) std::printf("%a: %a\n", x, got);
}

static void check(double x) {
    const float got = gmg::dw::narrow_sixth(x);
    const long double q = (long double)x / 6;
    ++checked;
    const long double top = std::ldexp((long double)1, 128) - std::ldexp((long double)1, 103);
    if (std::fabs(q) >= top * (1 + 1e-14L)) {  // beyond the last float's half step
        if (!std::isinf(got) || std::signbit(got) != std::signbit(x)) fail(x, got);
        return;
    }
    if (std::fabs(q) > top * (1 - 1e-14L)) return;  // either side of it
    int e;
    std::frexp(q, &e);  // |q| in [2^(e-1), 2^e)
    const bool sub = e - 1 < -126;
    const long double ulp = std::ldexp((long double)1, sub ? -149 : e - 1 - 23);
    const long double bound = ulp * (sub ? 0.75L : 0.5L + std::ldexp(1.0L, -21));
    // (a float past the top of the last binade is the next power of two)
    const long double v = std::isinf(got) ? std::copysign(std::ldexp((long double)1, 128), q) : got;
    if (!(std::fabs(v - q) <= bound)) fail(x, got);
}

int main() {
    std::mt19937_64 g(11);
    for (int e = 1023 - 155; e <= 1023 + 140; ++e)
        for (int k = 0; k < 20000; ++k) {
            const uint64_t frac = k == 0 ? 0 : k == 1 ? 0xfffffffffffffull : g() >> 12;
            for (int s = 0; s < 2; ++s)
                check(gmg::cvt::bits_d((uint64_t)s << 63 | (uint64_t)e << 52 | frac));
        }
    const double inf = std::numeric_limits<double>::infinity();
    for (double x : {inf, std::numeric_limits<double>::max(), 0x1p137, 0x1p500})
        for (double s : {1.0, -1.0}) {
            const float got = gmg::dw::narrow_sixth(s * x);
            if (!std::isinf(got) || std::signbit(got) != (s < 0)) fail(s * x, got);
        }
    for (double x : {0.0, -0.0}) {
        const float got = gmg::dw::narrow_sixth(x);
        if (got != 0 || std::signbit(got) != std::signbit(x)) fail(x, got);
    }
    for (double x : {std::numeric_limits<double>::denorm_min(), 1e-310, 1e-200})
        if (gmg::dw::narrow_sixth(x) != 0.f) fail(x, gmg::dw::narrow_sixth(x));
    if (!std::isnan(gmg::dw::narrow_sixth(std::nan("")))) fail(NAN, 0.f);
    std::printf("checked %lld, wrong %lld\n", checked, bad);
    return bad != 0;
}
