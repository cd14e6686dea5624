// npw_double.cuh -- double-precision arithmetic of the NPW_FP64 path with fewer FP64-pipe instructions and
// the same bits.
//
// The FP64 pipe of GB300 takes a warp instruction every 16 cycles per SM: one costs as much issue time
// as 64 float or integer ones, and comparisons count like adds.  So:
//   * A quotient n / x is the Markstein iteration (P. Markstein, IBM J. Res. Dev. 34(1), 1990): y
//     from the float reciprocal of x (2^-22) by one cubic step, nearly always 1 / x correctly rounded;
//     q0 = n y; q = q0 + (n - x q0) y with both operations fused, which is the correctly rounded quotient
//     but for divisors just below a power of two (see recip).  n - x q0 is exact because x lies in [2^-99,
//     2^99) and n is 0 or in [2^-872, 2^877).  Elsewhere the operator / is called, out of line.  Quotients
//     with one denominator share y: 3 FP64 instructions each after 3 for y, against about 9 for the operator.
//   * 2 c and 4 c and x / 4 are exact, so their products join the following sum in one fused
//     instruction that rounds as the sum alone.
//   * The monotone switch is decided in float from the exact-to-53-bits differences, with bounds that
//     also cover the rounding of the FP64 expressions; only what that does not decide evaluates them.
// tests/test_gpu_parity.py holds the results equal to the oracle, decisions and shape parameters bit
// for bit.
#pragma once
#include <cstdint>

#include "npw_bits.cuh"
#include "npw_internal.h"

namespace npw {
namespace f64 {

// y ~ 1 / x for the quotients below; false where x is outside [2^-99, 2^99) in magnitude
__device__ __forceinline__ bool recip_near(double x, double* y) {
    float xf;
    const bool ok = fast::seed_f(x, &xf);
    const double y0 = fast::widen_nz(fast::rcp_fast(xf));
    double e = fma(-x, y0, 1.0);
    e = fma(e, e, e);
    *y = fma(y0, e, y0);
    return ok;
}
// x whose mantissa begins with 13 ones, where the quotient with that y may be rounded wrongly.  With X, N the 53-bit
// integer mantissas, n / x lies c / (2 X) ulp from a rounding boundary, c a nonzero integer, and the quotient
// before its last rounding within |d eta| X 2^-105 ulp of n / x, d the error of n y rounded and eta that of y,
// both in ulps.  With d = 1/2 (at a boundary) a wrong rounding takes eta >= (2^53 / X)^2 / 2, and d = 3/2 takes
// eta N > 2^52 with N < X.  A correctly rounded y gives neither (Markstein's theorem); the cubic step leaves
// eta < 1/2 + 2^-15 for x near 2 (|1 - x y0| < 1.5 2^-23 there, cubed, and the last rounding), hence no wrong
// quotient below X = 2^53 (1 - 2^-14).
__device__ __forceinline__ bool hard(double x) { return (~(uint32_t)__double2hiint(x) & 0x000FFF80u) == 0u; }
// one Newton step: y correctly rounded, but where the mantissa of x is all ones (false)
__device__ __forceinline__ bool refine(double x, double* y) {
    *y = fma(fma(-x, *y, 1.0), *y, *y);
    return ((~(uint32_t)__double2hiint(x) & 0x000FFFFFu) | ~(uint32_t)__double2loint(x)) != 0u;
}
// 1 / x for quot: false outside the range and for hard x
__device__ __forceinline__ bool recip(double x, double* y) { return recip_near(x, y) & !hard(x); }
// n / x, y of recip(x), n in [2^-872, 2^877)
__device__ __forceinline__ double quot(double n, double x, double y) {
    const double q = n * y;
    return fma(fma(-x, q, n), y, q);
}
// the same with n = 0 allowed: the correction makes +0 of a -0, so the sign is taken from n y (one integer
// instruction)
__device__ __forceinline__ double quot0(double n, double x, double y) {
    const double q = n * y, r = fma(fma(-x, q, n), y, q);
    return __hiloint2double((__double2hiint(r) & 0x7FFFFFFF) | (__double2hiint(q) & (int)0x80000000), __double2loint(r));
}
__device__ __forceinline__ bool num_ok(double n) {
    const uint32_t h = (uint32_t)__double2hiint(n) & 0x7FFFFFFFu;
    return ((h >> 20) - 151u < 1749u) | ((h | (uint32_t)__double2loint(n)) == 0u);
}
static __device__ __noinline__ double div_any(double n, double x) { return n / x; }
__device__ __forceinline__ double div(double n, double x) {
    double y;
    const bool ok = recip(x, &y) & num_ok(n);
    return ok ? quot0(n, x, y) : div_any(n, x);
}

// n / x for n = 1/3 or 2/3: any x, hard ones too (the argument at weights_from, for the mantissa of 1/3)
__device__ __forceinline__ double div_third(double n, double x) {
    double y;
    return recip_near(x, &y) ? quot(n, x, y) : div_any(n, x);
}

// a truncated to float (0 where it is 0); *ok false outside [2^-99, 2^99)
__device__ __forceinline__ float to_f(double a, bool* ok) {
    float f;
    const bool in = fast::seed_f(a, &f);
    const bool zero = (((uint32_t)__double2hiint(a) & 0x7FFFFFFFu) | (uint32_t)__double2loint(a)) == 0u;
    *ok = *ok & (in | zero);
    return zero ? 0.0f : f;
}

}  // namespace f64

template <typename D>
__device__ __forceinline__ bool switch_fires(D w0, D w1, D w2, D w3, int variant);
template <typename D>
__device__ __forceinline__ bool k2_ratio_fires(D a, D b, D c);
static __device__ __noinline__ bool k2_ratio_fires_d(double a, double b, double c) { return k2_ratio_fires<double>(a, b, c); }
static __device__ __noinline__ bool switch_fires_d(double w0, double w1, double w2, double w3, int variant) {
    return switch_fires<double>(w0, w1, w2, w3, variant);
}

namespace f64 {

// Variant 0 of the monotone switch, as switch_fires<double> decides it.  d0, d1, d2: the neighbour
// differences in FP64, truncated to float (relative 2^-23); A, B, C of switch_v0_cert from them.  The
// errors against the exact quantities are those of the mixed path's level-2 test (fast::switch_level2)
// with twice the unit roundoff, plus 2^-52 |w| per difference; the FP64 expressions themselves are
// within 2^-44 (|w1| + |w2| + s) of the exact quantities in units of 12 p'.  e bounds all of it.
__device__ __forceinline__ bool switch_v0(double w0, double w1, double w2, double w3) {
    bool ok = true;
    const float d0 = to_f(w1 - w0, &ok), d1 = to_f(w2 - w1, &ok), d2 = to_f(w3 - w2, &ok);
    if (ok & (d0 == 0.0f) & (d1 == 0.0f) & (d2 == 0.0f)) return false;  // constant: every term is exactly 0
    const float m1 = to_f(w1, &ok), m2 = to_f(w2, &ok);
    const float t02 = d0 + d2, s = fabsf(d0) + fabsf(d2);
    const float A = fmaf(-2.f, d1, t02), B = d2 - d0, C = fmaf(14.f, d1, -t02);
    const float aA = fabsf(A), aB = fabsf(B), aC = fabsf(C);
    const float e = fmaf(0x1p-18f, s + aC, 0x1p-40f * (fabsf(m1) + fabsf(m2)));
    if (ok & (s < 0x1p60f) & (aC < 0x1p60f) & (s + aC > 0x1p-40f)) {
        const float E = fmaf(24.f, A, C), aE = fabsf(E), b12 = 12.f * aB, eE = 64.f * e;
        if (b12 > aE + eE) return true;
        if (aE > b12 + eE) {
            if (aB > fmaf(4.f, aA, 8.f * e)) return false;
            if ((aB < fmaf(4.f, aA, -8.f * e)) & (aA > e)) {
                const float G = fmaf(2.f * A, C, -3.f * B * B);
                if (fabsf(G) > 40.f * e * (aA + aB + aC + e)) return (G > 0.f) != ((A > 0.f) == (E > 0.f));
            }
        }
    }
    return switch_fires_d(w0, w1, w2, w3, 0);
}

// Table k3 shape parameter of the face with eta stencil w0..w3 and its flags, 0 where the switch, the guard
// or the bound says so (the guard is off by default in NPW_FP64)
__device__ __forceinline__ double face_eta(double w0, double w1, double w2, double w3, const MethodParams& mp, uint32_t* fl) {
    if (mp.scheme != NPW_RBF_ENO_ && mp.scheme != NPW_RBF_WENO_) return 0.0;
    if (mp.monotone_switch &&
        (mp.switch_variant == 0 ? switch_v0(w0, w1, w2, w3) : switch_fires_d(w0, w1, w2, w3, mp.switch_variant))) {
        *fl |= FL_SWITCH;
        return 0.0;
    }
    const double p1 = 15.0 * w1, p2 = 15.0 * w2;
    const double den0 = ((w0 - p1) + p2) - w3;
    if (mp.has_guard &&
        fabs(den0) <= mp.eta_guard * (((fabs(w0) + fabs(p1)) + fabs(p2)) + fabs(w3))) {
        *fl |= FL_ZERO_GUARD;
        return 0.0;
    }
    const double e = div(((w0 - 3.0 * w1) + 3.0 * w2) - w3, den0 + mp.eps_M);
    if (mp.has_bound && fabs(e) > mp.eta_max) {
        *fl |= FL_ZERO_BOUND;
        return 0.0;
    }
    return e;
}

// coefficients c_rj + q_rj eta of a face: rows 1 (k[0..2]) and 3 (k[3..5]); rows 2 and 0 mirror them
__device__ __forceinline__ void face_coefs(double eta, int rbf, double* k) {
    const bool ga = rbf == NPW_RBF_GA_;
    k[0] = 1.0 / 3.0 + (ga ? 2.0 / 3.0 : 5.0 / 6.0) * eta;
    k[1] = 5.0 / 6.0 + (ga ? -1.0 / 3.0 : -2.0 / 3.0) * eta;
    k[2] = -1.0 / 6.0 + (ga ? -1.0 / 3.0 : -1.0 / 6.0) * eta;
    k[3] = 1.0 / 3.0 + (ga ? 0.0 : -1.5) * eta;
    k[4] = -7.0 / 6.0 + (ga ? 3.0 : 6.0) * eta;
    k[5] = 11.0 / 6.0 + (ga ? -3.0 : -4.5) * eta;
}
// 0 + k0 x0 + k1 x1 + k2 x2 from the left (fma(k0, x0, 0) costs what the product does; the 0 counts where every
// product is -0)
__device__ __forceinline__ double dot(double k0, double x0, double k1, double x1, double k2, double x2) {
    return (fma(k0, x0, 0.0) + k1 * x1) + k2 * x2;
}

// WENO weights alpha_r / sum alpha of both sides from the squared denominators; false where a quotient
// may be wrong: outside the range of recip, or (REFINED: the mantissa all ones) for a hard sum.  The first
// quotients take any x: their dividends are the constants 0.1 and 0.3 (0.6), and a wrong one takes c = +-1, an X
// in the hard range that divides 2^53 N -+ 1 or 2^54 N -+ 1; none of these eight integers has a divisor there.
template <bool REFINED>
__device__ __forceinline__ bool weights_from(double x0, double x1, double x2, double wm[3], double wp[3]) {
    auto inv = [](double x, double* y) { return recip_near(x, y) & (REFINED ? refine(x, y) : !hard(x)); };
    double y0, y1, y2, ym, yp;
    bool ok = recip_near(x0, &y0);
    ok = recip_near(x1, &y1) & ok;
    ok = recip_near(x2, &y2) & ok;
    const double am0 = quot(0.3, x0, y0), ap0 = quot(0.1, x0, y0), a6 = quot(0.6, x1, y1), am2 = quot(0.1, x2, y2),
                 ap2 = quot(0.3, x2, y2);
    const double sm = (am0 + a6) + am2, sp = (ap0 + a6) + ap2;
    ok = inv(sm, &ym) & ok;
    ok = inv(sp, &yp) & ok;
    wm[0] = quot(am0, sm, ym);
    wm[1] = quot(a6, sm, ym);
    wm[2] = quot(am2, sm, ym);
    wp[0] = quot(ap0, sp, yp);
    wp[1] = quot(a6, sp, yp);
    wp[2] = quot(ap2, sp, yp);
    return ok;
}
// the rest, out of line: refined reciprocals (one cell in 4000 has a hard sum), else the operator /
static __device__ __noinline__ void weights_any(double x0, double x1, double x2, double wm[3], double wp[3]) {
    if (weights_from<true>(x0, x1, x2, wm, wp)) return;
    const double am[3] = {0.3 / x0, 0.6 / x1, 0.1 / x2}, ap[3] = {0.1 / x0, 0.6 / x1, 0.3 / x2};
    const double sm = (am[0] + am[1]) + am[2], sp = (ap[0] + ap[1]) + ap[2];
    for (int r = 0; r < 3; ++r) {
        wm[r] = am[r] / sm;
        wp[r] = ap[r] / sp;
    }
}

// Jiang-Shu weights of a cell (c = cells i-2..i+2), alpha_r / sum alpha of its right (wm) and left (wp)
// value from one set of indicators
__device__ __forceinline__ void cell_weights(const double* c, double eps_weno, double wm[3], double wp[3]) {
    const double t3 = 3.0 * c[2];
    const double a0 = fma(-2.0, c[3], c[2]) + c[4], b0 = fma(-4.0, c[3], t3) + c[4];
    const double a1 = fma(-2.0, c[2], c[1]) + c[3], b1 = c[1] - c[3];
    const double a2 = fma(-2.0, c[1], c[0]) + c[2], b2 = fma(-4.0, c[1], c[0]) + t3;
    double x0 = eps_weno + fma(0.25, b0 * b0, (13.0 / 12.0 * a0) * a0);
    double x1 = eps_weno + fma(0.25, b1 * b1, (13.0 / 12.0 * a1) * a1);
    double x2 = eps_weno + fma(0.25, b2 * b2, (13.0 / 12.0 * a2) * a2);
    x0 = x0 * x0;
    x1 = x1 * x1;
    x2 = x2 * x2;
    if (__builtin_expect(!weights_from<false>(x0, x1, x2, wm, wp), 0)) {
        double m[3], p[3];
        weights_any(x0, x1, x2, m, p);
        for (int r = 0; r < 3; ++r) {
            wm[r] = m[r];
            wp[r] = p[r];
        }
    }
}

// |a| < |b| and |a| > lim >= 0 by integer comparison (no FP64-pipe slot); NaN compares false
__device__ __forceinline__ uint64_t abs_bits(double a) { return (uint64_t)__double_as_longlong(a) & 0x7FFFFFFFFFFFFFFFull; }
__device__ __forceinline__ bool abs_less(double a, double b) {
    const uint64_t x = abs_bits(a), y = abs_bits(b);
    return (x < y) & (y <= 0x7FF0000000000000ull);
}
__device__ __forceinline__ bool abs_above(double a, double lim) {
    const uint64_t x = abs_bits(a);
    return (x > abs_bits(lim)) & (x <= 0x7FF0000000000000ull);
}

// eq. root_value on cells (a, b, c), den = -a + 2b - c as k2_ratio_fires forms it: 0 < num / den < 3.  The
// sign and the magnitude against 3 |den| are decided from both truncated to float (relative 2^-23
// each) where they are not within 2^-20 of the threshold, without the quotient.
__device__ __forceinline__ bool k2_switch(double a, double b, double c, double den) {
    const double num = fma(-2.0, a, 3.0 * b) - c;
    bool ok = true;
    const float n = to_f(num, &ok), d = to_f(den, &ok);
    if (ok) {
        if (n == 0.0f || d == 0.0f || (n > 0.0f) != (d > 0.0f)) return false;
        const float an = fabsf(n), ad = 3.0f * fabsf(d);
        if (an < ad * (1.0f - 0x1p-20f)) return true;
        if (an > ad * (1.0f + 0x1p-20f)) return false;
    }
    return k2_ratio_fires_d(a, b, c);
}

// Both shape parameters of one face value of a k = 2 cell, MQ: 2 num / (den + eps_M), Gaussian: half: a,
// b, d the cells beside, at and across from the face, t = -a + 2b - d.  On the 5-cell cross of Sec. 6 the
// numerator also carries the transverse second difference trans of the cell, with weight -1/4 for the
// stencil of the two cells at the face (central) and 1/8 for the extrapolating one: the terms that
// cancel the transverse curvature of the cell averages at the face midpoint.  Both share the
// denominator, hence its reciprocal.  need: bit 0 the central, bit 1 the extrapolating one is used;
// the other is formed only where it might reach the bound (its flag counts).
__device__ __forceinline__ void eta_k2_pair(double a, double b, double d, double t, double trans, int need,
                                            const MethodParams& mp, double* ec, double* ex, uint32_t* fl) {
    *ec = *ex = 0.0;
    const double den0 = fma(2.0, d, 5.0 * b - a);
    if (mp.has_guard && fabs(den0) <= mp.eta_guard * ((fabs(a) + 5.0 * fabs(b)) + 2.0 * fabs(d))) {
        *fl |= FL_ZERO_GUARD;
        return;
    }
    const double den = den0 + mp.eps_M;
    double y;
    const bool den_ok = recip(den, &y);
    const bool ga = mp.rbf == NPW_RBF_GA_;
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        if (x == 1 && trans == 0.0) {  // the same numerator
            *ex = *ec;
            break;
        }
        const double num = fma(x ? 0.125 : -0.25, trans, t);
        const bool used = ((need >> x) & 1) || (trans == 0.0);
        if (!used) {
            if (!mp.has_bound) continue;
            bool ok = true;
            const float n = to_f(num, &ok), m = to_f(den, &ok);
            if (ok && fabsf(n) * (ga ? 1.0f : 2.0f) < mp.eta_max_f * fabsf(m) * (1.0f - 0x1p-18f)) continue;
        }
        const double q = (den_ok & num_ok(num)) ? quot0(num, den, y) : div_any(num, den);
        double e = ga ? q : q + q;
        if (mp.has_bound && abs_above(e, mp.eta_max)) {
            *fl |= FL_ZERO_BOUND;
            e = 0.0;
        }
        *(x ? ex : ec) = e;
    }
}

}  // namespace f64
}  // namespace npw
