// tdist.h -- Student t critical values for the test of Eq. 7 (host, FP64).
#pragma once

namespace mcev {

// P(T <= t) for Student's t with integer nu >= 1 degrees of freedom.
double t_cdf_int(double t, int nu);
// t with P(T <= t) = p (0 < p < 1): rounded to FP32, the root that bisection of
// t_cdf_int ends at.
double t_quantile_int(double p, int nu);

}  // namespace mcev
