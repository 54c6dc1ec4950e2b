// The radial coordinate t = ln(r / r_k) / Delta of a spline segment, shared by the evaluation kernels.
#pragma once

#ifdef __CUDACC__
#include "nao_internal.h"

// log(1 + x) for the radial coordinate, x = r / r_k - 1, normally in [0, b), b = exp(Delta) - 1
// of the logarithmic grid. For |x| <= b <= 0.031 (grids with Delta <= 0.03) the Taylor series
// x - x^2/2 + x^3/3 - ... to x^12/12 (the first omitted term is below 2^-53 |x|), evaluated by
// Horner's rule; otherwise (coarser grids, r beyond the last knot) log1p.
__device__ __forceinline__ double log1p_small(double x, double b) {
    if (b > 0.031 || fabs(x) > b) return log1p(x);
    double p = -1.0 / 12.0;
    p = fma(p, x, 1.0 / 11.0);
    p = fma(p, x, -1.0 / 10.0);
    p = fma(p, x, 1.0 / 9.0);
    p = fma(p, x, -1.0 / 8.0);
    p = fma(p, x, 1.0 / 7.0);
    p = fma(p, x, -1.0 / 6.0);
    p = fma(p, x, 1.0 / 5.0);
    p = fma(p, x, -1.0 / 4.0);
    p = fma(p, x, 1.0 / 3.0);
    p = fma(p, x, -0.5);
    p = fma(p, x, 1.0);
    return p * x;
}

// Segment k and t in [0, 1) of rr = max(r, r0) in FP64: k from an FP32 logarithm, moved by one where it
// disagrees with the FP64 knots (r_k <= r < r_{k+1} as rr / r_k - 1 in [0, exp(Delta) - 1)), then
// t = log1p(rr / r_k - 1) / Delta.
__device__ __forceinline__ double radial_coordinate(const DevSystem &s, double rr, int &k) {
    const float sa = __logf((float)rr * (float)__ldg(s.inv_rk)) * (float)s.inv_delta;
    k = (int)floorf(sa);
    k = k < 0 ? 0 : (k > s.n_rgrid - 2 ? s.n_rgrid - 2 : k);
    double xr = fma(rr, __ldg(s.inv_rk + k), -1.0);
    if (xr < 0.0 && k > 0) {
        k--;
        xr = fma(rr, __ldg(s.inv_rk + k), -1.0);
    } else if (xr >= s.step_m1 && k < s.n_rgrid - 2) {
        k++;
        xr = fma(rr, __ldg(s.inv_rk + k), -1.0);
    }
    return log1p_small(xr, s.step_m1) * s.inv_delta;
}
#endif
