// x_rcp and x_rsqrt on the host with their FP32 estimates moved by up to two
// ulp either way: prints the largest relative error of each, in units of
// 2^-60, over the ends of the mantissa's range and random draws.
#include <cmath>
#include <cstdio>
#include <random>

#include "xf.cuh"

using namespace fpic;

static long double val(xf a)
{
    return std::ldexp((long double)a.m, a.e);
}

int main()
{
    std::mt19937_64 g(1);
    const long long lo = 0x2000000000000000ll, hi = 0x3fffffffffffffffll;
    long double worst[2] = {0, 0};
    for (int it = 0; it < 400000; ++it) {
        const int k = it & 3;
        const long long d = (long long)(g() >> (k < 2 ? 40 : 20));                // ends: 2^24, 2^44 units
        const long long m = k == 0 ? lo + d : k == 1 ? hi - d : k == 2 ? (it & 4 ? lo + d : hi - d)
                                                               : lo + (long long)(g() >> 3);
        const xf a = {m, -61 - (int)(g() % 4)};
        const long double x = val(a);
        const float y1 = 1.f / x_rcp_arg(a), y2 = (float)(1.0 / std::sqrt((double)x_rsqrt_arg(a)));
        for (int u = -2; u <= 2; ++u) {
            const auto move = [u](float y) { return x_float(x_float_bits(y) + (unsigned)u); };
            const long double e1 = std::fabs(val(x_rcp_est(a, move(y1))) * x - 1), r = val(x_rsqrt_est(a, move(y2)));
            const long double e2 = std::fabs(r * std::sqrt(x) - 1);
            worst[0] = std::fmax(worst[0], e1);
            worst[1] = std::fmax(worst[1], e2);
        }
    }
    for (int q = 0; q < 2; ++q) std::printf("%.3Lf\n", std::ldexp(worst[q], 60));
    return 0;
}
