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

#include <cmath>

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

// the same for any x > 0, infinity included
__device__ __forceinline__ double rcp64_inf(double x) { return __double2hiint(x) == 0x7ff00000 ? 0.0 : rcp64(x); }

// ---- FP32 base-2 logarithm and power: single MUFU instructions ------------

__device__ __forceinline__ float lg2_(float x) {
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float ex2_(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// ---- x^{-a} for a rational a = k / n with a small n (n = 0: pow) ----------
//
// u = x^{-1/n} from the FP32 MUFU and the binomial series to e^3. |e| stays below 4e-5
// (5e-6 in u at the ends of the range, from the logarithm, and 8e-6 where u is cut to
// 17 bits), so the next term stays below 2^-56. What remains are the roundings of the
// products. At n = 3 (p = 6 and 3) a u of 17 bits makes u^3 exact: two roundings, 1.08
// ulp at most (measured 1.00; 2.6 with all bits of u). Other n take u^k as u^n u^(k-n),
// since a rounding of u^n enters e too, with the weight -k/n: together -(k-n)/n of it is
// left (p = 4.5: measured 2.05 and 1.38 ulp, 2.9 and 2.6 with u^k by itself). pow, the
// other exponents' way, measured 1.2 ulp of its own, but of the rounded exponent, which
// adds |ln x| 2^-54 and more; the applies' errors against sums in extended precision are
// at or below its. 12 FP64 operations at n = 3 in place of about 100: A on 3 columns,
// 3,000 faces, 2.34 ms with pow, 0.79 ms; p = 4.5 0.92 ms.
struct RootPow {
    int n = 0, k = 0;
    float inv = 0.f;   // -1 / n
    double a = 0.0, c1 = 0.0, c2 = 0.0, c3 = 0.0;
};

// x^{-a}; *ix = 1/x. The conversions between FP32 and FP64 would run on the
// FP64 pipe: normal numbers are converted by shifting the bits instead (x
// truncated to FP32, which only moves the seed by 2^-23).
__device__ __forceinline__ double root_pow(double x, const RootPow& rp, double* ix) {
    const unsigned xh = (unsigned)__double2hiint(x), xl = (unsigned)__double2loint(x);
    // 2^-100 <= x < 2^100
    if (rp.n == 0 || xh - ((1023u - 100u) << 20) >= (200u << 20)) {
        *ix = rcp64_inf(x);
        return pow(x, -rp.a);
    }
    const float xf = __uint_as_float(__funnelshift_l(xl, xh, 3) - ((1023u - 127u) << 23));
    unsigned uf = __float_as_uint(ex2_(lg2_(xf) * rp.inv));
    if (rp.n == 3) uf = (uf + 0x40u) & ~0x7fu;   // 17 bits
    const double u = __hiloint2double((int)((uf >> 3) + ((1023u - 127u) << 20)), (int)(uf << 29));
    double un, uk;
    if (rp.n == 3) {   // k = 4 or 5: n = 3 for p = 6 and p = 3 alone
        const double u2 = u * u;
        un = u2 * u;
        uk = u2 * (rp.k == 5 ? un : u2);
    } else {
        double b = u, v = ((rp.k - rp.n) & 1) ? u : 1.0;
        un = (rp.n & 1) ? u : 1.0;
        for (int i = 1; rp.n >> i; ++i) {   // (k <= 2 n)
            b *= b;
            if ((rp.n >> i) & 1) un *= b;
            if (((rp.k - rp.n) >> i) & 1) v *= b;
        }
        uk = un * v;
    }
    const double e = fma(-x, un, 1.0);
    *ix = fma(un, fma(e, fma(e, e, e), e), un);
    return fma(uk * e, fma(fma(rp.c3, e, rp.c2), e, rp.c1), uk);
}

// the plan of |d|^{-2s}, s = 2 - 2/p (or, for L, of |d|^{-2(1 + 2/p)}): rational when
// 2 n / p is a whole number for some n <= 16 (p = 6: n = 3; 4.5: n = 9)
inline RootPow root_plan(double p, bool op_l) {
    RootPow r;
    const double q = 2.0 / p;
    r.a = op_l ? 3.0 - (2.0 - q) : 2.0 - q;
    for (int n = 1; n <= 16; ++n) {
        const double m = std::round(q * n);
        if (std::fabs(q * n - m) > 4e-16 * n) continue;
        const int k = op_l ? n + (int)m : 2 * n - (int)m;
        r.n = n;
        r.k = k;
        r.a = (double)k / n;
        r.inv = -1.f / (float)n;
        break;
    }
    r.c1 = r.a;
    r.c2 = 0.5 * r.a * (r.a + 1.0);
    r.c3 = r.a * (r.a + 1.0) * (r.a + 2.0) / 6.0;
    return r;
}

}  // namespace tp
