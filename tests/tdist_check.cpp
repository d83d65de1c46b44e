// Host check of the critical values (csrc/tdist.cpp): every value that enters a
// table (rounded to FP32) equals the root of the same CDF by plain bisection.
#include <cmath>
#include <cstdio>
#include <initializer_list>

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

int main() {
    const float alphas[] = {1e-6f, 0.0005f, 0.005f, 0.01f, 0.025f, 0.05f, 0.1f, 0.3f, 0.49f, 0.6f, 0.9f, 0.99f};
    long n = 0, bad = 0;
    for (const float a : alphas) {
        for (int nu = 1; nu <= 8191; nu += nu < 300 ? 1 : 97) {
            const double want = bisect(a, nu), got = mcev::t_quantile_int(a, nu);
            ++n;
            if ((float)want != (float)got && ++bad < 10) std::printf("alpha %g nu %d: %.17g != %.17g\n", a, nu, got, want);
        }
    }
    const double z = mcev::t_quantile_int(0.5, 40);
    if (!(std::fabs(z) < 1e-15)) ++bad;
    for (const double p : {0.0, 1.0, -1.0, std::nan("")})
        if (!std::isnan(mcev::t_quantile_int(p, 5))) ++bad;
    std::printf("%s %ld values, %ld differ\n", bad ? "FAIL" : "OK", n, bad);
    return bad ? 1 : 0;
}
