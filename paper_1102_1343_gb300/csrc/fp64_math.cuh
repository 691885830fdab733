// FP64 arithmetic of the right-hand side of eq. (F-disc).  This part issues
// FP64 instructions (compares, minima and conversions among them) at 1/64 of
// the FP32 rate, and the FP64 step is bound by that pipe (82 % busy, 9 % of
// the issue slots used).  So what can be done elsewhere is: signs, maxima and
// limits of non-negative numbers are taken on the bits by the integer units,
// square roots start from the hardware's approximation and take one step of
// third order, and the power comes from tables.  Measured, us per FP64 step,
// before and with this arithmetic (GB300): 2000^2 nodes (marching strips) 2318
// and 1635, 100^2 nodes (tiles) 62.4 and 53.7; with the adjoint of 510^2 nodes,
// 30 steps, 22.9 and 17.6 ms.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "fp64_tables.cuh"

namespace wf {

// The tests below are those of the comparisons that they stand for, with NaN
// counted as there: not above 0, not at most 0.  (Where only the upper word is
// looked at, x is the result of an operation and a NaN a quiet one.)

// x > 0 ? x : 0
__device__ __forceinline__ double pos64(double x) {
    return (unsigned)__double2hiint(x) <= 0x7ff00000u ? x : 0.0;
}
// the larger and the smaller of two numbers that are neither negative nor NaN
__device__ __forceinline__ double max_nn(double a, double b) {
    return (unsigned long long)__double_as_longlong(a) > (unsigned long long)__double_as_longlong(b) ? a : b;
}
__device__ __forceinline__ double min_nn(double a, double b) {
    return (unsigned long long)__double_as_longlong(a) < (unsigned long long)__double_as_longlong(b) ? a : b;
}
// x > 0
__device__ __forceinline__ bool gt0(double x) {
    return (unsigned long long)__double_as_longlong(x) - 1 < 0x7ff0000000000000ull;
}
// x at least 2^-1021 and finite
__device__ __forceinline__ bool normal64(double x) {
    return (unsigned)__double2hiint(x) - 0x00200000u < 0x7fd00000u;
}

// Roots and reciprocals by Householder's iteration (A. S. Householder, The
// Numerical Treatment of a Single Nonlinear Equation, 1970), one step of third
// order from the hardware's coarse approximation y (relative error below
// 2^-20).  1/sqrt(x): with e = 1 - x y^2 the value is y (1 - e)^(-1/2) =
// y (1 + e/2 + 3/8 e^2 + ...), what is left out is below 2^-58 and the error
// below 1.6 times 2^-53.  x is normal64.
__device__ __forceinline__ double rsqrt_seed(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return y;
}
__device__ __forceinline__ double rsqrt64(double x) {
    const double y = rsqrt_seed(x), e = fma(-(x * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}
// sqrt of x >= 0: with t = x y the value is t (1 - e)^(-1/2), e = 1 - t y
__device__ __forceinline__ double sqrt64(double x) {
    if (!normal64(x)) return sqrt(x);  // 0, subnormal, inf, NaN
    const double y = rsqrt_seed(x), t = x * y, e = fma(-t, y, 1.0);
    return fma(t * e, fma(0.375, e, 0.5), t);
}
// 1/x, 2^-1021 <= |x| < 2^1022 (a normal reciprocal): with e = 1 - x y the value
// is y/(1 - e) = y (1 + e + e^2 + ...); the error is below 1.1 times 2^-53
__device__ __forceinline__ double rcp64(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// x^b for a normal x > 0, |b log2 x| < 1000: 2^(b log2 x) by Tang's
// table-driven method (P. T. P. Tang, ACM TOMS 15 (1989) 144 and 16 (1990)
// 378).  x = 2^k m, m in [1, 2); r = c m - 1 with c the tabulated reciprocal
// of the middle of m's 128th, |r| < 2^-8; log2 x = (k + T) + (t + log2(1 + r))
// with k + T exact in 32 fractional bits, so that the product with b is
// rounded once.  2^y from the table of 2^(j/128) and a polynomial.  18 FP64
// operations; the error is below half of that of a rounded log2, product and
// exp2 (5.0e-15 against 9.8e-15 at worst over x from 1e-13 to 30, b from 0.9 to
// 2.2).
__device__ __forceinline__ double pow64(double x, double b) {
    const int hi = __double2hiint(x);
    const int i = (hi >> 13) & 127;
    const double2 ct = __ldg(reinterpret_cast<const double2 *>(kLogTab) + i);
    const double m = __hiloint2double((hi & 0x000fffff) | 0x3ff00000, __double2loint(x));
    const double r = fma(m, ct.x, -1.0);
    double q = fma(-0x1.ec709dc3a03fdp-3, r, 0x1.2776c50ef9bfep-2);
    q = fma(q, r, -0x1.71547652b82fep-2);
    q = fma(q, r, 0x1.ec709dc3a03fdp-2);
    q = fma(q, r, -0x1.71547652b82fep-1);
    q = fma(q, r, 0x1.71547652b82fep+0);
    const double l = fma(q, r, ct.y);
    // k + T: added to the bits of 1.5 2^20, whose last bit is 2^-32
    const double big = 0x1.8p+20;
    const long long kT = ((long long)((hi >> 20) - 1023) << 32) + (long long)__ldg(kLogInt + i);
    const double L = __longlong_as_double(__double_as_longlong(big) + kT) - big;
    const double y = fma(b, L, b * l);
    const double round = 0x1.8p+45;  // last bit 2^-7
    const double t = y + round;
    const int j = __double2loint(t);
    const double f = y - (t - round);
    double p = fma(0x1.5d87fe78a6731p-10, f, 0x1.3b2ab6fba4e77p-7);
    p = fma(p, f, 0x1.c6b08d704a0c0p-5);
    p = fma(p, f, 0x1.ebfbdff82c58fp-3);
    p = fma(p, f, 0x1.62e42fefa39efp-1);
    const double T = __ldg(kExpTab + (j & 127));
    const double v = fma(T, p * f, T);
    return __hiloint2double(__double2hiint(v) + ((j >> 7) << 20), __double2loint(v));
}
// a/b by the reciprocal and one correction with the exact residual (P. W.
// Markstein, IBM J. Res. Dev. 34 (1990) 111); divisors that have no normal
// reciprocal take the ordinary quotient
__device__ __forceinline__ double div64(double a, double b) {
    if (((unsigned)__double2hiint(b) & 0x7fffffffu) - 0x00200000u >= 0x7fb00000u) return a / b;
    const double y = rcp64(b), q = a * y;
    return fma(fma(-b, q, a), y, q);
}
// x^b of the capped wind component x >= 0: 0 where it is 0
__device__ __forceinline__ double wind_power64(double x, double b) {
    if (__double_as_longlong(x) == 0) return 0.0;
    const int hi = __double2hiint(x);
    // |b log2 x| < 900: x in [2^-64, 2^64) and b < 14 without a closer look
    if ((unsigned)(hi - 0x3bf00000) < 0x08000000u && __double2hiint(b) < 0x402c0000) return pow64(x, b);
    return exp2(b * log2(x));
}

// d, or 0 where it is at the rounding level of the difference of a and b,
// |d| <= 1e-9 (|a| + |b|).  Decided by the exponents wherever d's is less than
// 27 below the larger one's.
__device__ __forceinline__ double rounding_zero64(double d, double a, double b) {
    const int hd = __double2hiint(d) & 0x7fffffff;
    const int ha = __double2hiint(a) & 0x7fffffff, hb = __double2hiint(b) & 0x7fffffff;
    if (hd + (27 << 20) > (ha > hb ? ha : hb)) return d;
    return fabs(d) <= 1e-9 * (fabs(a) + fabs(b)) ? 0.0 : d;
}

// -F of eq. (F-disc) at a node (see neg_rhs2): some 40 FP64 operations and the
// power (95 in the form with IEEE square roots, fmax and exp2(b log2 x)).  On a
// mesh with dx = dy the differences are left in metres and 1/dx enters once.
template <bool HASM>
__device__ __forceinline__ double neg_rhs64(double p, double pl, double pr, double pd, double pu,
                                            double idx, double idy, double i2dx, double i2dy, double eps,
                                            double S0, double R0, double b, double c, double d, double e,
                                            double m, double un, double vn, double zx, double zy) {
    double xm = p - pl, xp = p - pr, ym = p - pd, yp = p - pu;
    double cx = rounding_zero64(pr - pl, pr, pl), cy = rounding_zero64(pu - pd, pu, pd);
    const bool iso = __double_as_longlong(idx) == __double_as_longlong(idy);
    if (!iso) {
        xm *= idx;
        xp *= idx;
        ym *= idy;
        yp *= idy;
        cx *= i2dx;
        cy *= i2dy;
    }
    const double gx = max_nn(pos64(xm), pos64(xp)), gy = max_nn(pos64(ym), pos64(yp));
    const double grad = sqrt64(fma(gx, gx, gy * gy));
    const double n2 = fma(cx, cx, cy * cy);
    const double rn = normal64(n2) ? rsqrt64(n2) : 0.0;
    const double U = fma(un, cx, vn * cy) * rn, tp = pos64(fma(zx, cx, zy * cy) * rn);
    const double pw = wind_power64(min_nn(pos64(U), e), b);
    // (R0 and c are negative for a moisture or a heat content without sense)
    const double s = max_nn(pos64(fma(d * tp, tp, fma(c, pw, R0))), S0);
    double S = HASM ? m * s : s;
    if (iso) S *= idx;
    const double nlap = (xm + xp) + (ym + yp);
    return S * fma(eps, nlap, grad);
}

}  // namespace wf
