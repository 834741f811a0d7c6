// FP64 division, square root and rational powers on the device in few operations of
// the FP64 pipe, which issues two lanes a cycle and SM and bounds every FP64 kernel.
//
// Each starts from an approximation of about 20 bits (rcp.approx.ftz.f64,
// rsqrt.approx.ftz.f64, or the FP32 MUFU) with a residual e that one fma gives almost
// exactly, and sums a series in e:
//   1 / x     = y / (1 - e),        e = 1 - x y:    y (1 + e + e^2 + e^3 + ..)
//   x^{-1/2}  = y (1 - e)^{-1/2},   e = 1 - x y^2:  y (1 + e/2 + 3 e^2/8 + ..)
//   x^{-a}    = u^k (1 - e)^{-a},   e = 1 - x u^n, a = k / n: the binomial series
// (geometric and binomial series: Abramowitz, Stegun, Handbook of Mathematical
// Functions, 3.6.8-3.6.10). A quotient or root is then corrected by its own residual,
// a - q b or x - s^2, which fma gives exactly (Markstein, Computation of elementary
// functions on the IBM RISC System/6000 processor, IBM J. Res. Dev. 34, 1990).
#pragma once

namespace tp {

// 1 / x for a normal x with a normal reciprocal: |e| < 2^-18, so the series stops
// below 2^-72 and the last rounding remains: 0.5 ulp (without the e^3 term 0.504)
__device__ __forceinline__ double rcp64(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, fma(e, e, e), e), y);
}
// a / b with r = rcp64(b): the rounded quotient, or the other neighbour where it lies
// within 2^-50 ulp of the middle of two numbers (b just below a power of two has such
// quotients); a result or residual below the normal range, and a zero's sign, are not
// kept so
__device__ __forceinline__ double div64(double a, double b, double r) {
    const double q = a * r;
    return fma(fma(-q, b, a), r, q);
}
// sqrt(x), rounded as div64 is, and its reciprocal in *r; x outside [1e-280, 1e280]
// takes the functions
__device__ __forceinline__ double sqrt64(double x, double* r) {
    if (!(x > 1e-280 && x < 1e280)) {
        const double s = sqrt(x);
        *r = 1.0 / s;
        return s;
    }
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x * y, y, 1.0);
    y = fma(y * e, fma(e, 0.375, 0.5), y);
    const double s0 = x * y;
    const double s = fma(fma(-s0, s0, x), 0.5 * y, s0);
    *r = fma(y, fma(-s, y, 1.0), y);
    return s;
}
__device__ __forceinline__ double third64(double x) { return div64(x, 3.0, 1.0 / 3.0); }

}  // namespace tp
