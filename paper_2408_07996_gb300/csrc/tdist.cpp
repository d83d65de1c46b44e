// tdist.cpp -- Student t distribution for integer degrees of freedom by the
// finite trigonometric series of Abramowitz & Stegun 26.7.3-26.7.4:
// with theta = atan(t / sqrt(nu)) and A(t|nu) = P(|T| <= t),
//   nu odd : A = (2/pi) (theta + sin(theta) (cos(theta) + 2/3 cos^3 + ...
//                 + (2*4*..*(nu-3)) / (1*3*..*(nu-2)) cos^(nu-2)))   (nu > 1)
//            A = 2 theta / pi                                         (nu = 1)
//   nu even: A = sin(theta) (1 + 1/2 cos^2 + 1*3/(2*4) cos^4 + ...
//                 + (1*3*..*(nu-3)) / (2*4*..*(nu-2)) cos^(nu-2))
// All terms are positive, so the sum is stable in FP64 for the nu <= 2^16
// the renderer needs.  The critical value of the one-tailed test (Sec. 3.2)
// is the alpha-quantile of that CDF, rounded to FP32: Newton steps from the
// expansion of the quantile in 1/nu (A&S 26.7.5), kept inside a bracket.  Where the
// series' rounding leaves room for more than one FP32 value (small alpha, large
// nu), the value is the one that bisection of the computed CDF ends at, so the tables
// hold bisection's values for every alpha.  The series costs nu/2 divisions in a
// chain, so the number of its evaluations is what the table costs: 2 to 4 per
// value instead of about 60 by bisection alone (on an x86 host, alpha 0.05 and 0.01:
// a 15-value table up to nu = 255 0.13 -> 0.01 ms, 128 values up to 8191 21 -> 0.4
// ms; alpha 1e-6 2.3 ms, 1e-12 11 ms).
#include "tdist.h"

#include <algorithm>
#include <cmath>

namespace mcev {

static double abs_prob(double t, int nu) {
    const double th = std::atan(std::fabs(t) / std::sqrt((double)nu));
    const double c = std::cos(th), s = std::sin(th), c2 = c * c;
    if (nu % 2 == 1) {
        if (nu == 1) return 2.0 * th / M_PI;
        double term = c, sum = c;
        for (int k = 1; 2 * k + 1 <= nu - 2; ++k) {
            term *= c2 * (2.0 * k) / (2.0 * k + 1.0);
            sum += term;
        }
        return 2.0 / M_PI * (th + s * sum);
    }
    double term = 1.0, sum = 1.0;
    for (int k = 1; 2 * k <= nu - 2; ++k) {
        term *= c2 * (2.0 * k - 1.0) / (2.0 * k);
        sum += term;
    }
    return s * sum;
}

double t_cdf_int(double t, int nu) {
    if (std::isnan(t)) return t;
    if (std::isinf(t)) return t > 0 ? 1.0 : 0.0;
    const double a = abs_prob(t, nu);
    return t >= 0.0 ? 0.5 * (1.0 + a) : 0.5 * (1.0 - a);
}

// p-quantile of the standard normal distribution, to the accuracy a starting
// point needs: Newton steps on erfc
static double normal_quantile(double p) {
    const bool upper = p > 0.5;
    const double q = upper ? 1.0 - p : p;
    double z = -std::sqrt(std::max(0.0, -2.0 * std::log(2.0 * q)));   // P(Z <= z) <= exp(-z^2/2)/2
    for (int it = 0; it < 50; ++it) {
        const double f = 0.5 * std::erfc(-z * M_SQRT1_2) - q;
        const double step = f / (std::exp(-0.5 * z * z) / std::sqrt(2.0 * M_PI));
        z -= step;
        if (std::fabs(step) < 1e-12 * (1.0 + std::fabs(z))) break;
    }
    return upper ? -z : z;
}

// The quantile by bisection of the computed CDF.  [a, b] holds every root that the
// series' rounding allows: outside it the CDF lies on the side of p that the
// position tells, so it is evaluated inside only.  Stops when both ends round to
// the same FP32 value, which is what the tables hold.
static double bisect(double p, int nu, double a, double b) {
    auto cdf = [&](double t) { return t < a ? 0.0 : (t > b ? 1.0 : t_cdf_int(t, nu)); };
    double lo = -1.0, hi = 1.0;
    while (cdf(lo) > p) lo *= 2.0;
    while (cdf(hi) < p) hi *= 2.0;
    for (int it = 0; it < 200 && (float)lo != (float)hi; ++it) {
        const double mid = 0.5 * (lo + hi);
        if (mid == lo || mid == hi) break;
        if (cdf(mid) < p) lo = mid;
        else hi = mid;
    }
    return 0.5 * (lo + hi);
}

double t_quantile_int(double p, int nu) {
    if (!(p > 0.0 && p < 1.0)) return std::nan("");
    // What rounding makes of the CDF: at most about 2 nu + 16 units of 2^-53 (every
    // term of the series is a product of up to nu / 2 factors), taken twice.  A p of
    // that size has no root worth the name, only the one that bisection ends at.
    const double noise = (4.0 * nu + 32.0) * 0x1p-53;
    if (std::min(p, 1.0 - p) < 64.0 * noise) return bisect(p, nu, -HUGE_VAL, HUGE_VAL);
    const double z = normal_quantile(p), z2 = z * z, v = 1.0 / nu;
    const double g1 = z * (z2 + 1.0) / 4.0;
    const double g2 = z * ((5.0 * z2 + 16.0) * z2 + 3.0) / 96.0;
    const double g3 = z * (((3.0 * z2 + 19.0) * z2 + 17.0) * z2 - 15.0) / 384.0;
    const double g4 = z * ((((79.0 * z2 + 776.0) * z2 + 1482.0) * z2 - 1920.0) * z2 - 945.0) / 92160.0;
    double t = z + v * (g1 + v * (g2 + v * (g3 + v * g4)));
    // log of the density's constant
    const double lc = std::lgamma(0.5 * (nu + 1.0)) - std::lgamma(0.5 * nu) - 0.5 * std::log(nu * M_PI);
    double lo = -HUGE_VAL, hi = HUGE_VAL;     // cdf(lo) < p <= cdf(hi)
    for (int it = 0; it < 100; ++it) {
        const double f = t_cdf_int(t, nu) - p;
        const double pdf = std::exp(lc - 0.5 * (nu + 1.0) * std::log1p(t * t / nu));
        const double step = f / pdf;
        if (std::fabs(step) <= 1e-9 * std::fabs(t) || std::fabs(f) <= noise) {
            // a Newton step of this size leaves an error below the CDF's own rounding
            t -= step;
            const double range = 2.0 * noise / pdf + 1e-15 * std::fabs(t);
            if ((float)(t - range) == (float)(t + range)) return t;
            // (the density must not fall off within the range)
            if (range * (nu + 1.0) * std::fabs(t) < 0.1 * (nu + t * t)) return bisect(p, nu, t - range, t + range);
            break;
        }
        if (f < 0.0) lo = t;
        else hi = t;
        double next = t - step;
        if (!(next > lo && next < hi)) {
            // outside the bracket (or no density left): halve it, or widen it
            if (std::isinf(lo)) next = hi > 0.0 ? -1.0 : 2.0 * hi - 1.0;
            else if (std::isinf(hi)) next = lo < 0.0 ? 1.0 : 2.0 * lo + 1.0;
            else next = 0.5 * (lo + hi);
            if (next == lo || next == hi) break;
        }
        t = next;
    }
    return bisect(p, nu, -HUGE_VAL, HUGE_VAL);
}

}  // namespace mcev
