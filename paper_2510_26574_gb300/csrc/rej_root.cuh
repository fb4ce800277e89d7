// Square root and quotient of Algorithm 3's steps (factor.cu): a column of H over
// sqrt(H(i,i)), with one reciprocal root for both, 11 dependent FP64 operations instead of ~20.
#pragma once

namespace kevd {

// s = sqrt(h) and y = 1 / sqrt(h) for normal h: Halley's iteration on a reciprocal-root
// estimate (relative error below 2^-22, cubed), then one correction of s = h y by its exact
// residual (P. Markstein, IBM J. Res. Dev. 34(1), 1990).
__device__ __forceinline__ void rej_root(double h, double& s, double& y) {
    double y0;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y0) : "d"(h));
    const double e = fma(-(h * y0), y0, 1.0);
    y = fma(fma(e, 0.375, 0.5), y0 * e, y0);
    const double s0 = h * y;
    s = fma(fma(-s0, s0, h), 0.5 * y, s0);
}

// c / s, y = 1 / s up to rounding: the quotient corrected by its exact residual (as above).
__device__ __forceinline__ double rej_quot(double c, double s, double y) {
    const double q = c * y;
    return fma(fma(-q, s, c), y, q);
}

}  // namespace kevd
