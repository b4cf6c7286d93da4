// FP64 functions of few operations: GB300 issues about two FP64 operations an
// SM and clock, so their number is the cost of the kernels that call these.
#pragma once

namespace pbg {

// 1/b from the hardware's approximation y (rcp.approx.ftz.f64, whose operand and
// result have 20 fraction bits) and one step of the hyperpower iteration of order
// three (M. Altman, Pacific J. Math. 10 (1960) 1107): with e = 1 - b y,
// 1/b = y / (1 - e) = y (1 + e + e^2 + O(e^3)), and e^3 is below 2^-55.
// Four FP64 operations.  For b of 2^-1000 to 2^1000.
__device__ __forceinline__ double rcp_fp64(double b) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
    const double e = fma(-b, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// 1/sqrt(a), a >= 0, from the hardware's approximation y (rsqrt.approx.ftz.f64, whose
// operand and result have 20 fraction bits) and one step of third order (A. S.
// Householder, The Numerical Treatment of a Single Nonlinear Equation, 1970):
// with e = 1 - a y^2, 1/sqrt(a) = y (1 - e)^(-1/2) = y (1 + e/2 + 3 e^2/8 + O(e^3)),
// and e^3 is below 2^-54, its term 5/16 of that.  Five FP64 operations.
// (Starting from rsqrtf costs two conversions, which are FP64-rate too: 140
// against 121 us for the pair sum of 2,000 atoms with the library's function.)
// Zero, subnormal arguments and infinity take the library's function.
__device__ __forceinline__ double rsqrt_fp64(double a) {
    if ((unsigned)__double2hiint(a) - 0x00100000u >= 0x7fe00000u) return rsqrt(a);
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
    const double e = fma(-(a * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

// exp(-u) for u >= 0, by argument reduction and a table (W. J. Cody and W.
// Waite, Software Manual for the Elementary Functions, 1980; P. T. P. Tang,
// ACM TOMS 15 (1989) 144): -u = (n/64) ln 2 + f, |f| <= ln 2 / 128, the Taylor
// polynomial of degree 5 of exp(f) (its remainder f^6/720 is below 4e-17), and
// 2^(n/64) from tab, the 64 values 2^(i/64), and an exponent.  ln 2 / 64 in two
// parts keeps f exact to rounding.  Ten FP64 operations.  Zero from u = 708 on,
// where exp(-u) is 3.3e-308 (decided on u's upper word, an integer comparison:
// n below is a 32-bit number and would wrap from u = 2.3e7 on).
__device__ __forceinline__ double exp_neg_fp64(double u, const double *tab) {
    constexpr double MAGIC = 6755399441055744.0;  // 1.5 * 2^52: rounds to an integer
    constexpr double HI = 0x1.62e42fefa39efp-7, LO = 0x1.abc9e3b39803fp-62;
    const double t = fma(u, -92.332482616893656, MAGIC);
    const int n = __double2loint(t);
    const double nd = t - MAGIC;
    const double f = fma(nd, -LO, fma(nd, -HI, -u));
    double p = 1.0 / 120.0;
    p = fma(p, f, 1.0 / 24.0);
    p = fma(p, f, 1.0 / 6.0);
    p = fma(p, f, 0.5);
    p = fma(p, f, 1.0);
    p = fma(p, f, 1.0);
    const double v = p * tab[n & 63];
    const double r = __hiloint2double(__double2hiint(v) + (n >> 6) * 1048576, __double2loint(v));
    return __double2hiint(u) >= 0x40862000 ? 0.0 : r;  // 708.0
}

}  // namespace pbg
