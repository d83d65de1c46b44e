// Host check of the critical values (csrc/tdist.cpp) over every alpha the entry
// points take, down to FP32 denormals and up to the last value below 1: rounded to
// FP32, each equals the root that bisection of the same CDF ends at.
#include <cmath>
#include <cstdio>
#include <initializer_list>
#include <random>

#include "tdist.h"

static double bisect(double p, int nu) {
    double lo = -1.0, hi = 1.0;
    while (mcev::t_cdf_int(lo, nu) > p) lo *= 2.0;
    while (mcev::t_cdf_int(hi, nu) < p) hi *= 2.0;
    for (int it = 0; it < 200; ++it) {
        const double mid = 0.5 * (lo + hi);
        if (mid == lo || mid == hi) break;
        if (mcev::t_cdf_int(mid, nu) < p) lo = mid;
        else hi = mid;
    }
    return 0.5 * (lo + hi);
}

static long n = 0, bad = 0;
static void check(double p, int nu) {
    const double want = bisect(p, nu), got = mcev::t_quantile_int(p, nu);
    ++n;
    if ((float)want != (float)got && ++bad < 10) std::printf("p %g nu %d: %.17g != %.17g\n", p, nu, got, want);
}

int main() {
    for (const float a : {1e-45f, 1e-40f, 1e-30f, 1e-20f, 1e-16f, 1e-15f, 1e-14f, 1e-12f, 1e-10f, 1e-9f, 1e-8f, 1e-7f,
                          0.4999999f, 0.5f, 0.5000001f, 0.999f, 0.999999f, 0.99999994f})
        for (const int nu : {1, 2, 3, 4, 5, 7, 10, 15, 16, 31, 63, 100, 255, 511, 1023, 4095, 16383}) {
            check(a, nu);
            check(0.5 * (double)a, nu);   // the two-tailed test's
        }
    std::mt19937_64 g(3);
    std::uniform_real_distribution<double> u(0.0, 1.0);
    for (int i = 0; i < 20000; ++i) {
        const int nu = (int)std::exp(u(g) * std::log(8192.0));
        const double e = std::exp(-100.0 * u(g) * u(g));
        const float a = (float)(i % 3 ? e : 1.0 - e);
        if (a > 0.0f && a < 1.0f) check(i % 2 ? a : 0.5 * (double)a, nu);
    }
    std::printf("%s %ld values, %ld differ\n", bad ? "FAIL" : "OK", n, bad);
    return bad ? 1 : 0;
}
