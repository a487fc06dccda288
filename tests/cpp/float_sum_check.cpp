// The three-float running sum (paper_2302_07084_gb300/csrc/float_sum.h, the code the
// Hessian sums run) against exact integer sums: terms are integers below 2^24 times
// powers of two, so sums are exact in 128 bits. Compiled without contraction. Bound:
// the value's rounding, 2^-53 of the sum, and n^3 / 6 2^-72 of the terms' sizes (see the
// header). A pair of floats (hi + lo) has to miss the bound somewhere, or the terms are
// too easy. Prints "ok".
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <random>

#include "float_sum.h"

int main() {
    std::mt19937_64 rng(7);
    int pair_misses = 0;
    double worst = 0, worst64 = 0;
    for (int kind = 0; kind < 4; ++kind)   // one sign and size, one sign, both signs, cancelling
        for (int n : {1, 2, 3, 40, 41, 128, 500, 1500})
            for (int rep = 0; rep < 200; ++rep) {
                lne::FloatSum s = {0.f, 0.f, 0.f};
                float phi = 0.f, plo = 0.f;
                double d = 0.0, size = 0.0;
                __int128 exact = 0;
                float last = 0.f;
                for (int i = 0; i < n; ++i) {
                    int64_t m = (int64_t)(rng() & 0xFFFFFF);
                    const int e = kind == 0 ? 10 : (int)(rng() % 28);
                    if (kind >= 2 && (rng() & 1)) m = -m;
                    float p = std::ldexp((float)m, e);
                    if (kind == 3 && (i & 1)) p = -last + std::ldexp((float)(m & 0xFF), 0);
                    last = p;
                    exact += (__int128)(int64_t)p;
                    size += std::fabs((double)p);
                    lne::float_sum_add(s, p);
                    float err;
                    phi = lne::two_sum(phi, p, &err);
                    plo += err;
                    d += (double)p;
                }
                const double unit = std::ldexp(1.0, -53), sum = std::fabs((double)exact);
                const double bound = sum * unit + (double)n * n * n / 6.0 * std::ldexp(1.0, -72) * size;
                auto off = [&](double v) {
                    const __int128 t = (__int128)v - exact;
                    return (double)(t < 0 ? -t : t);
                };
                const double e3 = off(lne::float_sum_value(s)), e2 = off((double)phi + (double)plo), e64 = off(d);
                if (e3 > bound * (1.0 + 1e-9)) {
                    std::printf("kind %d n %d: off by %g, bound %g\n", kind, n, e3, bound);
                    return 1;
                }
                pair_misses += e2 > bound * (1.0 + 1e-9);
                worst = std::fmax(worst, e3 / size);
                worst64 = std::fmax(worst64, e64 / size);
            }
    std::printf("largest error over the terms' sizes: three floats %.3g, FP64 %.3g; pairs beyond the bound: %d\n", worst,
                worst64, pair_misses);
    if (pair_misses == 0 || worst > worst64) return 1;
    std::printf("ok\n");
    return 0;
}
