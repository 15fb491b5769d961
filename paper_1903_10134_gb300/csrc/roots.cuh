// Square root and its reciprocal from an estimate of the reciprocal, by Newton's
// iteration in fused multiply-adds, for kernels that need both and for which a correctly
// rounded root and quotient cost too much.  Usable on the host too: a test there checks
// the bounds below for every estimate within the hardware's stated error.
#pragma once

#include <cmath>

#include "f64bits.cuh"

namespace mdpd {

MDPD_HD float fma_t(float a, float b, float c) { return fmaf(a, b, c); }
MDPD_HD double fma_t(double a, double b, double c) { return fma(a, b, c); }

// 1 / sqrt(x) from an estimate y within 2 ulp: within 1 ulp, half of it from the last
// rounding and half from that of x y (the iteration's own error is 1.5 e^2 for an
// estimate off by e, some 1e-13 in FP32).
template <typename T>
MDPD_HD T inv_sqrt_step(T x, T y)
{
    return fma_t(T(0.5) * y, fma_t(-x * y, y, T(1)), y);
}

// sqrt(x) from y = 1 / sqrt(x) within 1 ulp: x y with its error, whose fused residual is
// exact, taken back.  Within 0.500001 ulp, so correctly rounded but for near ties.
template <typename T>
MDPD_HD T sqrt_from(T x, T y)
{
    const T r = x * y;
    return fma_t(T(0.5) * y, fma_t(-r, r, x), r);
}

}  // namespace mdpd
