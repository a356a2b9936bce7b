// pdq_lf_math.cuh -- the FP64 root and exponential of the 1-D Eulerian model's march, from the hardware's
// estimates (rsqrt_seed, rcp_seed: relative error below 2^-19) and the mathematics given at each.
#pragma once

#include "pdq_device.cuh"

namespace pdq {

// The root u > 0 of g(u) = u^2/2 + a u - c = 0, a > 0, c > 0: the chord method (simplified Newton), whose fixed
// slope is known beforehand.  g'(u) = u + a, which at the root is s = sqrt(a^2 + 2c), so y, the estimate of 1/s, serves
// as 1/g' and no division is refined.  With y = (1 + d)/s a step u <- u - y g(u) takes a relative error e to
// -e (d + (1 + d) e u/(2s)), u <= s.  The start 2c / (a + s), from two estimates, has e <= 2^-18; one step leaves
// 2^-36, the second 2^-55.  The rounding of u/2 + a enters as 2^-53 c y <= 2^-53 u.
__device__ __forceinline__ double lf_root(double a, double c) {
    const double cc = c + c, x = __fma_rn(a, a, cc), y = rsqrt_seed(x);
    double u = cc * rcp_seed(__fma_rn(x, y, a));
    u = __fma_rn(-y, __fma_rn(u, __fma_rn(0.5, u, a), -c), u);
    return __fma_rn(-y, __fma_rn(u, __fma_rn(0.5, u, a), -c), u);
}

// (e^x - 1)/x and E = e^x for x <= 0: above -1/2 the Taylor polynomial, to x^6/7! while |x| < 2^-6 (half of the march's
// cells; truncation below x^7/8! = 2^-57), else to x^14/15! (truncation below 2^-15/16! = 2^-59); from -1/2 on the library's
// exponential, and the quotient by iterative refinement: q <- q + r (em - x q) with r the estimate of 1/x takes
// q's relative error from d to d^2 to d^3 <= 2^-57.
__device__ __forceinline__ double lf_phi64(double x, double* E) {
    if (x > -0.5) {
        double p = 1.0 / 5040.0;
        if (x <= -0.015625) {
            p = 1.0 / 1307674368000.0;                            // 1/15!
            p = __fma_rn(p, x, 1.0 / 87178291200.0);
            p = __fma_rn(p, x, 1.0 / 6227020800.0);
            p = __fma_rn(p, x, 1.0 / 479001600.0);
            p = __fma_rn(p, x, 1.0 / 39916800.0);
            p = __fma_rn(p, x, 1.0 / 3628800.0);
            p = __fma_rn(p, x, 1.0 / 362880.0);
            p = __fma_rn(p, x, 1.0 / 40320.0);
            p = __fma_rn(p, x, 1.0 / 5040.0);
        }
        p = __fma_rn(p, x, 1.0 / 720.0);
        p = __fma_rn(p, x, 1.0 / 120.0);
        p = __fma_rn(p, x, 1.0 / 24.0);
        p = __fma_rn(p, x, 1.0 / 6.0);
        p = __fma_rn(p, x, 0.5);
        p = __fma_rn(p, x, 1.0);
        *E = __fma_rn(x, p, 1.0);
        return p;
    }
    *E = exp(x);
    const double em = *E - 1.0, r = rcp_seed(x);
    double q = em * r;
    q = __fma_rn(__fma_rn(-x, q, em), r, q);
    return __fma_rn(__fma_rn(-x, q, em), r, q);
}

}  // namespace pdq
