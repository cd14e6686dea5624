// npw_device.cuh -- per-face arithmetic of the non-polynomial ENO3 / WENO5 method on the GPU.
//
// R is the state type (double or float); D is the type in which the shape parameter, the
// monotone switch, the ENO choice and the smoothness indicators are evaluated (double).
// In the double instantiation every expression is written in a fixed evaluation order and
// the translation unit is compiled without multiply-add contraction, so that results are
// reproducible bit for bit from the cell averages.
//
// Paper passages: Sec. 2 (stencils S_r(i), v^{(r)-}_{i+1/2} = sum_j c_rj vbar_{i-r+j}, eq.
// weno_re with alpha_r = d_r / (eps + beta_r)^2), Sec. 3.5 Table k3 (coefficients and eta;
// row r = -1 uses 11/6), Sec. 3.3 (Gaussian recipe; k = 3 rows derived from the flat limit of
// the Gaussian interpolant of the primitive), Sec. 4 (eq. root_value, eq. adaptation),
// Sec. 5.1 (Lax-Friedrichs flux), Sec. 5.2 Ex. 4 (Euler, ideal gas).  k = 2: Sec. 3.2-3.5
// Table k2 with the shape parameter of eq. i+1/2_eps_approx (MQ) / i+1/2_eps_approx1
// (Gaussian), the Gaussian rows r = -1, 1 from the flat limit, and the switch of eq.
// root_value / eq. adaptation on the cell's three-cell stencil.
#pragma once
#include <cstdint>

#include "npw_double.cuh"
#include "npw_internal.h"

namespace npw {

// n / x: the operator, or in double its correctly rounded form with fewer FP64 instructions
__device__ __forceinline__ float quotient(float n, float x) { return n / x; }
__device__ __forceinline__ double quotient(double n, double x) { return f64::div(n, x); }


// ---------------------------------------------------------------------------------------
// Table k3.  row = r + 1 for r = -1..2; row r gives the value at face x_{i+1/2} from the
// cells i-r, i-r+1, i-r+2.
// ---------------------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ T poly_coef(int row, int j) {
    switch (row * 3 + j) {
        case 0: return T(11.0 / 6.0);
        case 1: return T(-7.0 / 6.0);
        case 2: return T(1.0 / 3.0);
        case 3: return T(1.0 / 3.0);
        case 4: return T(5.0 / 6.0);
        case 5: return T(-1.0 / 6.0);
        case 6: return T(-1.0 / 6.0);
        case 7: return T(5.0 / 6.0);
        case 8: return T(1.0 / 3.0);
        case 9: return T(1.0 / 3.0);
        case 10: return T(-7.0 / 6.0);
        default: return T(11.0 / 6.0);
    }
}

// coefficient of eta: multiquadric (Table k3, right) or Gaussian (Sec. 3.3 recipe, k = 3)
template <typename T>
__device__ __forceinline__ T pert_coef(int rbf, int row, int j) {
    if (rbf == NPW_RBF_GA_) {
        switch (row * 3 + j) {
            case 0: return T(-3.0);
            case 1: return T(3.0);
            case 2: return T(0.0);
            case 3: return T(2.0 / 3.0);
            case 4: return T(-1.0 / 3.0);
            case 5: return T(-1.0 / 3.0);
            case 6: return T(-1.0 / 3.0);
            case 7: return T(-1.0 / 3.0);
            case 8: return T(2.0 / 3.0);
            case 9: return T(0.0);
            case 10: return T(3.0);
            default: return T(-3.0);
        }
    }
    switch (row * 3 + j) {
        case 0: return T(-9.0 / 2.0);
        case 1: return T(6.0);
        case 2: return T(-3.0 / 2.0);
        case 3: return T(5.0 / 6.0);
        case 4: return T(-2.0 / 3.0);
        case 5: return T(-1.0 / 6.0);
        case 6: return T(-1.0 / 6.0);
        case 7: return T(-2.0 / 3.0);
        case 8: return T(5.0 / 6.0);
        case 9: return T(-3.0 / 2.0);
        case 10: return T(6.0);
        default: return T(-9.0 / 2.0);
    }
}

// ---------------------------------------------------------------------------------------
// Shape parameter (Table k3): eta = (w0 - 3 w1 + 3 w2 - w3) / (w0 - 15 w1 + 15 w2 - w3 + eps_M)
// with w = cells i-1..i+2 of face i+1/2.
// ---------------------------------------------------------------------------------------
template <typename D>
__device__ __forceinline__ D eta_num(D w0, D w1, D w2, D w3) {
    return w0 - D(3.0) * w1 + D(3.0) * w2 - w3;
}
template <typename D>
__device__ __forceinline__ D eta_den(D w0, D w1, D w2, D w3) {
    return w0 - D(15.0) * w1 + D(15.0) * w2 - w3;
}

// ---------------------------------------------------------------------------------------
// Monotone switch (Sec. 4).
// Variant 0: the cubic p with averages w0..w3 over the cells of the eta stencil, in
// s = (x - x_{i+1/2})/dx on -2 < s < 2; 12 p'(s) = A s^2 + B s + C with
//   A = 6 ((w3 - w0) + 3 (w1 - w2)),  B = 6 ((w0 - w1) + (w3 - w2)),
//   C = (w0 - w3) + 15 (w2 - w1).
// p is non-monotone iff 12 p' takes both signs on the open interval: min < 0 < max over
// 12p'(-2) = 4A - 2B + C, 12p'(2) = 4A + 2B + C and, when the vertex -B/(2A) is strictly
// inside (|B| < 4|A|), 12p'(vertex) = C - B^2/(4A).
// Variant 1: the k = 2 ratio of eq. root_value on cells (w0, w1, w2) and on (w1, w2, w3).
// ---------------------------------------------------------------------------------------
template <typename D>
__device__ __forceinline__ bool k2_ratio_fires(D a, D b, D c) {
    D num = D(-2.0) * a + D(3.0) * b - c;
    D den = -a + D(2.0) * b - c;
    if (den == D(0.0)) return false;
    D ratio = num / den;
    return ratio > D(0.0) && ratio < D(3.0);
}

template <typename D>
__device__ __forceinline__ bool switch_fires(D w0, D w1, D w2, D w3, int variant) {
    if (variant == 1) {
        bool f1 = k2_ratio_fires(w0, w1, w2);
        bool f2 = k2_ratio_fires(w1, w2, w3);
        return f1 || f2;
    }
    D A = D(6.0) * ((w3 - w0) + D(3.0) * (w1 - w2));
    D B = D(6.0) * ((w0 - w1) + (w3 - w2));
    D C = (w0 - w3) + D(15.0) * (w2 - w1);
    D vm = D(4.0) * A - D(2.0) * B + C;
    D vp = D(4.0) * A + D(2.0) * B + C;
    D mn = vm < vp ? vm : vp;
    D mx = vm < vp ? vp : vm;
    if (A != D(0.0) && fabs(B) < D(4.0) * fabs(A)) {
        D vv = C - B * B / (D(4.0) * A);
        mn = vv < mn ? vv : mn;
        mx = vv > mx ? vv : mx;
    }
    return mn < D(0.0) && mx > D(0.0);
}

// ---------------------------------------------------------------------------------------
// ENO stencil choice from Newton divided differences (Sec. 2, Sec. 3.1): c0..c4 = cells
// i-2..i+2; the left extension is taken only when strictly smaller.  Returns r.
// ---------------------------------------------------------------------------------------
template <typename D>
__device__ __forceinline__ int eno_choice(D c0, D c1, D c2, D c3, D c4) {
    D dl = fabs(c2 - c1);
    D dr = fabs(c3 - c2);
    if (dl < dr) {
        D ddl = fabs(c0 - D(2.0) * c1 + c2);
        D ddr = fabs(c1 - D(2.0) * c2 + c3);
        return (ddl < ddr) ? 2 : 1;
    }
    D ddl = fabs(c1 - D(2.0) * c2 + c3);
    D ddr = fabs(c2 - D(2.0) * c3 + c4);
    return (ddl < ddr) ? 1 : 0;
}

// ---------------------------------------------------------------------------------------
// k = 2.  Table k2: row = r + 1 for r = -1, 0, 1; row r gives the value at x_{i+1/2} from the
// cells i-r, i-r+1.  A cell i has the stencil c[0..2] = cells i-1, i, i+1; its two face
// values use their own shape parameters (side 0: v^-_{i+1/2}; side 1: v^+_{i-1/2}, the mirror).
// ---------------------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ T poly2_coef(int row, int j) {
    switch (row * 2 + j) {
        case 0: return T(3.0 / 2.0);
        case 1: return T(-1.0 / 2.0);
        case 2: return T(1.0 / 2.0);
        case 3: return T(1.0 / 2.0);
        case 4: return T(-1.0 / 2.0);
        default: return T(3.0 / 2.0);
    }
}

// coefficient of eta: multiquadric (Table k2, right) or Gaussian (r = 0: eq. i+1/2_approx1;
// r = -1, 1: flat limit of the Gaussian interpolant)
template <typename T>
__device__ __forceinline__ T pert2_coef(int rbf, int row, int j) {
    if (rbf == NPW_RBF_GA_) {
        switch (row * 2 + j) {
            case 0: return T(-2.0);
            case 1: return T(0.0);
            case 2: return T(1.0 / 2.0);
            case 3: return T(1.0 / 2.0);
            case 4: return T(0.0);
            default: return T(-2.0);
        }
    }
    switch (row * 2 + j) {
        case 0: return T(-3.0 / 2.0);
        case 1: return T(1.0 / 2.0);
        case 2: return T(1.0 / 4.0);
        case 3: return T(1.0 / 4.0);
        case 4: return T(1.0 / 2.0);
        default: return T(-3.0 / 2.0);
    }
}

// WENO3 linear weights: v^-_{i+1/2} d = (2/3, 1/3) for r = 0 (cells i, i+1), r = 1 (i-1, i);
// v^+_{i-1/2} mirrored
template <typename T>
__device__ __forceinline__ T lin_weight2(int side, int r) {
    if (side == 0) return r == 0 ? T(2.0 / 3.0) : T(1.0 / 3.0);
    return r == 0 ? T(1.0 / 3.0) : T(2.0 / 3.0);
}

// value of cell i at its right (side 0) or left (side 1) face, k = 2; c[0..2] = cells i-1..i+1;
// eta_c: shape parameter of the central row (row 0), eta_x: of the extrapolating rows
// shift (points off the face midpoint, Sec. 6): the transverse term sigma sy, added to each
// candidate; the midpoint passes none
template <typename R, typename D>
__device__ __forceinline__ R cell_face_value_k2(const R* c, int side, R eta_c, R eta_x, const MethodParams& mp,
                                               int* r_out, R shift = R(0.0), bool shifted = false) {
    R cand[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int row = (side == 0) ? r : r - 1;
        const R eta = row == 0 ? eta_c : eta_x;
        R s = R(0.0);
#pragma unroll
        for (int j = 0; j < 2; ++j) s += (poly2_coef<R>(row + 1, j) + pert2_coef<R>(mp.rbf, row + 1, j) * eta) * c[1 - r + j];
        cand[r] = shifted ? s + shift : s;
    }
    if (mp.scheme == NPW_ENO_ || mp.scheme == NPW_RBF_ENO_) {
        const int r = fabs(D(c[1]) - D(c[0])) < fabs(D(c[2]) - D(c[1])) ? 1 : 0;
        *r_out = r;
        return cand[r];
    }
    *r_out = 0;
    const D b0 = (D(c[2]) - D(c[1])) * (D(c[2]) - D(c[1]));
    const D b1 = (D(c[1]) - D(c[0])) * (D(c[1]) - D(c[0]));
    const R den0 = R(D(mp.eps_weno) + b0), den1 = R(D(mp.eps_weno) + b1);
    const R a0 = lin_weight2<R>(side, 0) / (den0 * den0);
    const R a1 = lin_weight2<R>(side, 1) / (den1 * den1);
    R asum = R(0.0);
    asum += a0;
    asum += a1;
    R v = R(0.0);
    v += (a0 / asum) * cand[0];
    v += (a1 / asum) * cand[1];
    return v;
}

// value of a k = 2 cell as cell_face_value_k2<double> gives it (no shift): the ENO candidate alone, or
// the WENO3 mean with one reciprocal per denominator
__device__ __forceinline__ double cell_value_k2_d(const double* c, int side, double eta_c, double eta_x, int r,
                                                  const MethodParams& mp) {
    const bool ga = mp.rbf == NPW_RBF_GA_;
    auto cand = [&](int q) {
        const int row = side == 0 ? q : q - 1;
        const double eta = row == 0 ? eta_c : eta_x;
        // rows -1 (3/2, -1/2), 0 (1/2, 1/2), 1 (-1/2, 3/2) with their perturbations
        const double p0 = row == 0 ? 0.5 : (row < 0 ? 1.5 : -0.5), p1 = row == 0 ? 0.5 : (row < 0 ? -0.5 : 1.5);
        const double far_ = ga ? -2.0 : -1.5, near_ = ga ? 0.0 : 0.5, mid = ga ? 0.5 : 0.25;
        const double q0 = row == 0 ? mid : (row < 0 ? far_ : near_), q1 = row == 0 ? mid : (row < 0 ? near_ : far_);
        return fma(p0 + q0 * eta, c[1 - q], 0.0) + (p1 + q1 * eta) * c[2 - q];  // (as f64::dot)
    };
    if (mp.scheme == NPW_ENO_ || mp.scheme == NPW_RBF_ENO_) return r == 0 ? cand(0) : cand(1);
    const double g0 = c[2] - c[1], g1 = c[1] - c[0];
    double x0 = mp.eps_weno + g0 * g0, x1 = mp.eps_weno + g1 * g1;
    x0 = x0 * x0;
    x1 = x1 * x1;
    const double a0 = f64::div_third(side == 0 ? 2.0 / 3.0 : 1.0 / 3.0, x0), a1 = f64::div_third(side == 0 ? 1.0 / 3.0 : 2.0 / 3.0, x1);
    const double sum = a0 + a1;
    return fma(f64::div(a0, sum), cand(0), 0.0) + f64::div(a1, sum) * cand(1);
}

// One field at one face, k = 2.  w[0..5] = cells i-2..i+3 around face i+1/2; v^- from cell i
// (stencil w[1..3]), v^+ from cell i+1 (stencil w[2..4]); tl, tr: transverse second
// differences of cells i and i+1 (0 on a line).  Flag bits: 0 switch of cell i, 3 switch of
// cell i+1, 2 / 4 ENO r of cell i / i+1, 6 / 7 an eta of v^- zeroed by the guard / the bound,
// 8 / 9 the same for v^+.
// Arithmetic of npw_double.cuh; eta of v^- and v^+ from f64::eta_k2_pair.
__device__ __forceinline__ uint32_t face_field_k2_d(const double* w, const MethodParams& mp, double* vm, double* vp,
                                                    double tl, double tr, double* eta_out) {
    uint32_t fl = 0;
    const bool eno = mp.scheme == NPW_ENO_ || mp.scheme == NPW_RBF_ENO_;
    int rl = 0, rr = 0;
    if (eno) {
        const double d0 = w[2] - w[1], d1 = w[3] - w[2], d2 = w[4] - w[3];
        rl = f64::abs_less(d0, d1) ? 1 : 0;
        rr = f64::abs_less(d1, d2) ? 1 : 0;
    }
    double el = 0.0, er = 0.0, elx = 0.0, erx = 0.0;
    if (mp.scheme == NPW_RBF_ENO_ || mp.scheme == NPW_RBF_WENO_) {
        // -a + 2b - c of either cell, the switch's denominator and the numerator of v^- of the left cell
        const double sl = fma(2.0, w[2], -w[1]) - w[3], sr = fma(2.0, w[3], -w[2]) - w[4];
        // v^-: r = 0 the central row, 1 the extrapolating one; v^+: the other way round (eta_out: central)
        const int need_l = eno && !eta_out ? (rl == 0 ? 1 : 2) : 3, need_r = eno ? (rr == 1 ? 1 : 2) : 3;
        if (mp.monotone_switch && f64::k2_switch(w[1], w[2], w[3], sl))
            fl |= FL_SWITCH;
        else
            f64::eta_k2_pair(w[1], w[2], w[3], sl, tl, need_l, mp, &el, &elx, &fl);
        if (mp.monotone_switch && f64::k2_switch(w[2], w[3], w[4], sr)) {
            fl |= FL_SWITCH_R_K2;
        } else {
            uint32_t zr = 0;
            f64::eta_k2_pair(w[4], w[3], w[2], fma(2.0, w[3], -w[4]) - w[2], tr, need_r, mp, &er, &erx, &zr);
            fl |= zr << 2;  // FL_ZERO_GUARD_R_K2, FL_ZERO_BOUND_R_K2
        }
    }
    *vm = cell_value_k2_d(w + 1, 0, el, elx, rl, mp);
    *vp = cell_value_k2_d(w + 2, 1, er, erx, rr, mp);
    fl |= (uint32_t(rl & 1) << 2) | (uint32_t(rr & 1) << 4);
    if (eta_out) *eta_out = el;
    return fl;
}

// ---------------------------------------------------------------------------------------
// k = 2 on the 5-cell cross at a point of the face (Sec. 6; the two Gauss points of eq.
// 2DIntegral, Sec. 7): the 3-cell stencil of the two cells of the ENO row along the normal and
// the transverse neighbour that ENO picks, evaluated sigma cell widths from the face midpoint,
// is the Table k2 row plus sigma times the one-sided transverse difference sy toward that
// neighbour (side sg = +1 / -1).  Its Taylor error there is e v_xx dx^2 + (1/24 + sg sigma/2 -
// sigma^2/2) v_yy dy^2 - (sigma/2) v_xy dx dy (e = 1/6 for the two cells at the face, -1/3 for
// the extrapolating pair, whose perturbation weights sum to -2 times the central row's), and the
// shape parameter cancels it: numerator -a2 + t trans + x xy, central t = -1/4 + 3 sigma^2 -
// 3 sg sigma, x = 3 sigma; extrapolating t = 1/8 - 3/2 sigma^2 + 3/2 sg sigma, x = -3/2 sigma;
// xy is the mixed difference of the cell with the cell across the face on the sg side.
// ---------------------------------------------------------------------------------------
template <typename D>
struct CrossSide {
    D trans, sg, sy, xy;  // of one cell of the face: second difference, ENO side, one-sided difference, mixed
};

// transverse data of a cell from its column (lo, c, hi across the line) and, for xy, the cell
// across the face (alo, a, ahi) on the same rows
template <typename D>
__device__ __forceinline__ CrossSide<D> cross_side(D lo, D c, D hi, D alo, D a, D ahi) {
    CrossSide<D> cs;
    const D dn = c - lo, up = hi - c;
    cs.trans = (lo - D(2.0) * c) + hi;
    const bool lower = fabs(dn) < fabs(up);
    cs.sg = lower ? D(-1.0) : D(1.0);
    cs.sy = lower ? dn : up;
    cs.xy = lower ? -((alo - lo) - (a - c)) : ((ahi - hi) - (a - c));
    return cs;
}

template <typename D>
__device__ __forceinline__ D eta_k2_point(const D* c, int side, bool central, const CrossSide<D>& cs, D sigma,
                                          const MethodParams& mp, uint32_t* zr) {
    const D a = side == 0 ? c[0] : c[2];
    const D b = c[1];
    const D d = side == 0 ? c[2] : c[0];
    const D s = cs.sg;
    const D t_tr = central ? (D(-0.25) + D(3.0) * sigma * sigma) - D(3.0) * s * sigma
                           : (D(0.125) - D(1.5) * sigma * sigma) + D(1.5) * s * sigma;
    const D t_xy = central ? D(3.0) * sigma : D(-1.5) * sigma;
    const D num = ((-a + D(2.0) * b - d) + t_tr * cs.trans) + t_xy * cs.xy;
    const D den0 = -a + D(5.0) * b + D(2.0) * d;
    const D mag = fabs(a) + D(5.0) * fabs(b) + D(2.0) * fabs(d);
    if (mp.eta_guard > 0.0 && fabs(den0) <= D(mp.eta_guard) * mag) {
        *zr |= FL_ZERO_GUARD;
        return D(0.0);
    }
    const D e = (mp.rbf == NPW_RBF_GA_ ? D(1.0) : D(2.0)) * num / (den0 + D(mp.eps_M));
    if (mp.eta_max > 0.0 && fabs(e) > D(mp.eta_max)) {
        *zr |= FL_ZERO_BOUND;
        return D(0.0);
    }
    return e;
}

// One field at one point of a face (sigma from its midpoint), k = 2 on the cross: as
// face_field_k2, with l / r the transverse data of the cells behind v^- / v^+.
template <typename R, typename D>
__device__ __forceinline__ uint32_t face_point_k2(const R* w, const MethodParams& mp, R* vm, R* vp,
                                                  const CrossSide<D>& l, const CrossSide<D>& r, D sigma) {
    uint32_t fl = 0;
    R el = R(0.0), er = R(0.0), elx = R(0.0), erx = R(0.0);
    if (mp.scheme == NPW_RBF_ENO_ || mp.scheme == NPW_RBF_WENO_) {
        const D cl[3] = {D(w[1]), D(w[2]), D(w[3])};
        const D cr[3] = {D(w[2]), D(w[3]), D(w[4])};
        if (mp.monotone_switch && k2_ratio_fires<D>(cl[0], cl[1], cl[2])) {
            fl |= FL_SWITCH;
        } else {
            el = R(eta_k2_point<D>(cl, 0, true, l, sigma, mp, &fl));
            elx = R(eta_k2_point<D>(cl, 0, false, l, sigma, mp, &fl));
        }
        if (mp.monotone_switch && k2_ratio_fires<D>(cr[0], cr[1], cr[2])) {
            fl |= FL_SWITCH_R_K2;
        } else {
            uint32_t zr = 0;
            er = R(eta_k2_point<D>(cr, 1, true, r, sigma, mp, &zr));
            erx = R(eta_k2_point<D>(cr, 1, false, r, sigma, mp, &zr));
            fl |= zr << 2;  // FL_ZERO_GUARD_R_K2, FL_ZERO_BOUND_R_K2
        }
    }
    int rl = 0, rr = 0;
    *vm = cell_face_value_k2<R, D>(w + 1, 0, el, elx, mp, &rl, R(sigma * l.sy), true);
    *vp = cell_face_value_k2<R, D>(w + 2, 1, er, erx, mp, &rr, R(sigma * r.sy), true);
    fl |= (uint32_t(rl & 1) << 2) | (uint32_t(rr & 1) << 4);
    return fl;
}

// One field at one face, k = 3 (arguments and flags as face_field): the weights of both cells, the
// coefficients once; arithmetic of npw_double.cuh
__device__ __forceinline__ uint32_t face_field_d(const double* w, const MethodParams& mp, double* vm, double* vp,
                                                 double* eta_out) {
    uint32_t fl = 0;
    const double eta = f64::face_eta(w[1], w[2], w[3], w[4], mp, &fl);
    if (eta_out) *eta_out = eta;
    double k[6];
    f64::face_coefs(eta, mp.rbf, k);
    const double m0 = f64::dot(k[0], w[2], k[1], w[3], k[2], w[4]), m1 = f64::dot(k[2], w[1], k[1], w[2], k[0], w[3]),
                 m2 = f64::dot(k[3], w[0], k[4], w[1], k[5], w[2]);
    const double p0 = f64::dot(k[5], w[3], k[4], w[4], k[3], w[5]), p1 = f64::dot(k[0], w[2], k[1], w[3], k[2], w[4]),
                 p2 = f64::dot(k[2], w[1], k[1], w[2], k[0], w[3]);
    if (mp.scheme == NPW_ENO_ || mp.scheme == NPW_RBF_ENO_) {
        const int rl = eno_choice<double>(w[0], w[1], w[2], w[3], w[4]), rr = eno_choice<double>(w[1], w[2], w[3], w[4], w[5]);
        *vm = rl == 0 ? m0 : (rl == 1 ? m1 : m2);
        *vp = rr == 0 ? p0 : (rr == 1 ? p1 : p2);
        return fl | (uint32_t(rl & 3) << 2) | (uint32_t(rr & 3) << 4);
    }
    double a[3], b[3], unused[3];
    f64::cell_weights(w, mp.eps_weno, a, unused);
    f64::cell_weights(w + 1, mp.eps_weno, unused, b);
    *vm = f64::dot(a[0], m0, a[1], m1, a[2], m2);
    *vp = f64::dot(b[0], p0, b[1], p1, b[2], p2);
    return fl;
}

// One field at one face.  w[0..5] = cells i-2..i+3 around face i+1/2.  Returns the flag
// byte (bit0 switch, bits 2-3 / 4-5 ENO r of the left / right cell, bit 6 / 7 the evaluated eta
// zeroed by the guard / the bound).
// eta_out (may be NULL): the face's shape parameter as used (k = 2: that of v^-, central row)
__device__ __forceinline__ uint32_t face_field(const double* w, const MethodParams& mp, double* vm, double* vp, double tl = 0.0,
                                               double tr = 0.0, double* eta_out = nullptr) {
    return mp.k == 2 ? face_field_k2_d(w, mp, vm, vp, tl, tr, eta_out) : face_field_d(w, mp, vm, vp, eta_out);
}

// ---------------------------------------------------------------------------------------
// Near ties of the threshold decisions at one face (the FL_NEAR_TIE bit of npweno_reconstruct):
// a quantity that decides the monotone switch, the guard or the bound lies within tol
// (relative) of its threshold, so that two correct evaluations in different forms (the
// switch's closed form here, an elimination elsewhere; the guard in float or in double) may
// decide differently.  The ENO choice is not among them: it compares two differences of the
// same cell averages, which every correct evaluation rounds alike, so it is expected to agree
// everywhere.  Margins (all in double, from the cell averages):
//   switch variant 0 (Sec. 4, the cubic on the eta stencil): 12 p' at either end or at an
//     inside vertex within 8 tol (|w0| + .. + |w3|) of 0 (times 12), or the vertex within
//     8 tol of an end of the stencil;  the ratio test (variant 1, k = 2): its denominator
//     within tol (|a| + |b| + |c|) of 0, or the ratio within 4 tol of 0 or 3;  a stencil of
//     equal averages is constant, hence monotone, and not a tie;
//   guard: |den| within tol of the guard threshold; bound: |eta| within tol of eta_max.
// w[0..5] = cells i-2..i+3 of face i+1/2.
// ---------------------------------------------------------------------------------------
// two exactly equal zeros (a plateau) compare the same way in any evaluation: not a tie
__device__ __forceinline__ bool tie_rel(double a, double b, double tol) {
    const double m = fmax(fabs(a), fabs(b));
    return m > 0.0 && fabs(a - b) <= tol * m;
}
__device__ __forceinline__ bool k2_ratio_near(double a, double b, double c, double tol) {
    if (a == b && b == c) return false;  // constant stencil: monotone, decided exactly
    const double num = -2.0 * a + 3.0 * b - c, den = -a + 2.0 * b - c;
    if (fabs(den) <= tol * (fabs(a) + fabs(b) + fabs(c))) return true;
    if (den == 0.0) return false;
    const double r = num / den;
    return fabs(r) <= 4.0 * tol || fabs(r - 3.0) <= 4.0 * tol;
}
__device__ __forceinline__ bool switch_v0_near(const double* w, double tol) {
    if (w[0] == w[1] && w[1] == w[2] && w[2] == w[3]) return false;  // constant stencil
    const double A = 6.0 * ((w[3] - w[0]) + 3.0 * (w[1] - w[2]));
    const double B = 6.0 * ((w[0] - w[1]) + (w[3] - w[2]));
    const double C = (w[0] - w[3]) + 15.0 * (w[2] - w[1]);
    const double lim = 12.0 * 8.0 * tol * (fabs(w[0]) + fabs(w[1]) + fabs(w[2]) + fabs(w[3]));
    bool near = fabs(4.0 * A - 2.0 * B + C) <= lim || fabs(4.0 * A + 2.0 * B + C) <= lim;
    if (A != 0.0) {
        const double sv = -B / (2.0 * A);
        near = near || fabs(fabs(sv) - 2.0) <= 8.0 * tol;
        if (fabs(sv) < 2.0) near = near || fabs(C - B * B / (4.0 * A)) <= lim;
    }
    return near;
}
// near tie of a k = 2 face of the RBF schemes, in double; w[1..4] = cells i-1..i+2
__device__ __forceinline__ bool face_near_tie_k2(const double* w, const MethodParams& mp, double tol) {
    bool near = false;
    if (mp.monotone_switch) near = k2_ratio_near(w[1], w[2], w[3], tol) || k2_ratio_near(w[2], w[3], w[4], tol);
    for (int side = 0; side < 2; ++side) {
        const double* c = w + 1 + side;  // cell i (side 0, v^-) or i + 1 (side 1, v^+)
        const double a = side == 0 ? c[0] : c[2], b = c[1], d = side == 0 ? c[2] : c[0];
        const double den0 = -a + 5.0 * b + 2.0 * d, mag = fabs(a) + 5.0 * fabs(b) + 2.0 * fabs(d);
        if (mp.eta_guard > 0.0) near = near || tie_rel(fabs(den0), mp.eta_guard * mag, tol);
        if (mp.eta_max > 0.0) {
            const double e = (mp.rbf == NPW_RBF_GA_ ? 1.0 : 2.0) * (-a + 2.0 * b - d) / (den0 + mp.eps_M);
            near = near || tie_rel(fabs(e), mp.eta_max, tol);
        }
    }
    return near;
}
static __device__ __noinline__ bool face_near_tie_d(double w1, double w2, double w3, double w4, const MethodParams& mp,
                                                    double tol) {
    const double w[6] = {0.0, w1, w2, w3, w4, 0.0};  // (both orders use cells i-1..i+2)
    const bool rbf = mp.scheme == NPW_RBF_ENO_ || mp.scheme == NPW_RBF_WENO_;
    bool near = false;
    if (mp.k == 2) {
        if (rbf) near = face_near_tie_k2(w, mp, tol);
        return near;
    }
    if (rbf && mp.monotone_switch)
        near = near || (mp.switch_variant == 1 ? (k2_ratio_near(w[1], w[2], w[3], tol) || k2_ratio_near(w[2], w[3], w[4], tol))
                                               : switch_v0_near(w + 1, tol));
    if (rbf) {
        const double den0 = eta_den<double>(w[1], w[2], w[3], w[4]);
        const double mag = fabs(w[1]) + 15.0 * fabs(w[2]) + 15.0 * fabs(w[3]) + fabs(w[4]);
        if (mp.eta_guard > 0.0) near = near || tie_rel(fabs(den0), mp.eta_guard * mag, tol);
        if (mp.eta_max > 0.0)
            near = near || tie_rel(fabs(eta_num<double>(w[1], w[2], w[3], w[4]) / (den0 + mp.eps_M)), mp.eta_max, tol);
    }
    return near;
}

// Certainly no near tie at a k = 3 face (switch variant 0), in float: every quantity compared by
// face_near_tie lies further from its threshold than tol and the bounds here together.  A, B, C of
// switch_v0_cert from the neighbour differences truncated or rounded to float, e bounds their errors (as
// in fast::switch_level2, f64::switch_v0; a sixty-fourth of that of E = 24 A + C).  Nearly every face
// passes; the rest takes the FP64 expressions, some 60 FP64-pipe instructions, which bounded
// npweno_reconstruct before.
__device__ __forceinline__ bool far_from_ties(float d0, float d1, float d2, float a1, float a2, float unit, float abs_err,
                                              const MethodParams& mp, float tol, bool exact_ab = false) {
    const float t02 = d0 + d2, s = fabsf(d0) + fabsf(d2);
    const float A = fmaf(-2.f, d1, t02), B = d2 - d0, C = fmaf(14.f, d1, -t02);
    const float aA = fabsf(A), aB = fabsf(B), aC = fabsf(C);
    const float e = fmaf(unit, s + aC, abs_err * (a1 + a2));
    const float mag = 2.f * (a1 + a2) + s;  // at least |w0| + .. + |w3|
    if (!((s < 0x1p50f) & (aC < 0x1p50f) & (s + aC > 0x1p-40f))) return false;
    bool far_ = true;
    if (mp.monotone_switch) {
        const float lim = 100.f * tol * mag, E = fmaf(24.f, A, C), aE = fabsf(E), eE = fmaf(64.f, e, lim), b12 = 12.f * aB;
        far_ = fabsf(b12 - aE) > eE + 0x1p-20f * (b12 + aE);  // both ends
        const float a4 = 4.f * aA, e8 = exact_ab ? 0.0f : 8.f * e;
        const bool inside = aB < a4 * (1.f - 0x1p-10f) - e8,
                   outside = aB > fmaf(a4, 1.f + 0x1p-10f, e8) || (exact_ab && aA == 0.0f);
        const float G = fmaf(2.f * A, C, -3.f * B * B);
        far_ = far_ & (outside | (inside & (fabsf(G) > fmaf(40.f * e, aA + aB + aC + e, 2.5f * aA * lim))));
    }
    if (mp.has_guard) {
        const float g = mp.eta_guard_f * (fabsf(a1) * 16.f + fabsf(a2) * 16.f);  // (the magnitudes, within s + ...)
        const float gm = mp.eta_guard_f * s;
        far_ = far_ & ((aC > g * 1.01f + 2.f * gm + 64.f * e) | (aC < g * 0.85f - 2.f * gm - 64.f * e));
    }
    if (mp.has_bound) {
        const float x = mp.eta_max_f * aC, m = fmaf(mp.eta_max_f, fabsf(mp.eps_M_f) + 64.f * e, 64.f * e);
        far_ = far_ & (fabsf(aA - x) > 0x1p-10f * (aA + x) + m);
    }
    return far_;
}

// K2: float data of order k = 2, known at compile time
template <typename R, bool K2>
__device__ __forceinline__ bool face_near_tie(const R* wr, const MethodParams& mp, double tol) {
    if (!K2 && mp.k == 3 && (mp.scheme == NPW_RBF_ENO_ || mp.scheme == NPW_RBF_WENO_) && mp.guard_switch && mp.tie_tol_f <= 0x1p-14f) {
        // a constant stencil: monotone; its denominator and numerator against positive thresholds are exactly 0 in
        // float (15 w is exact in double) and where w = 0, but round-off of 15 w and 3 w in double
        if (wr[1] == wr[2] && wr[2] == wr[3] && wr[3] == wr[4] &&
            (sizeof(R) == sizeof(float) || wr[1] == R(0.0) || (!mp.has_guard && !mp.has_bound)))
            return false;
        bool ok = true;
        if constexpr (sizeof(R) == sizeof(float)) {
            const float d0 = wr[2] - wr[1], d1 = wr[3] - wr[2], d2 = wr[4] - wr[3];
            ok = far_from_ties(d0, d1, d2, fabsf(wr[2]), fabsf(wr[3]), 0x1p-19f, 0.0f, mp, mp.tie_tol_f);
            if (!ok) {
                // nearly linear data: A and B are a few units of round-off, but then exact.  A difference is
                // exact where adding it back gives the other cell, either way round.
                const float t02 = d0 + d2, A = fmaf(-2.f, d1, t02), B = d2 - d0;
                auto sum_exact = [](float x, float y, float z) { return z - x == y && z - y == x; };
                if (sum_exact(wr[2], -wr[1], d0) && sum_exact(wr[3], -wr[2], d1) && sum_exact(wr[4], -wr[3], d2) &&
                    sum_exact(d0, d2, t02) && sum_exact(t02, -2.f * d1, A) && sum_exact(d2, -d0, B))
                    ok = far_from_ties(d0, d1, d2, fabsf(wr[2]), fabsf(wr[3]), 0x1p-19f, 0.0f, mp, mp.tie_tol_f, true);
            }
        } else {
            const float d0 = f64::to_f(wr[2] - wr[1], &ok), d1 = f64::to_f(wr[3] - wr[2], &ok),
                        d2 = f64::to_f(wr[4] - wr[3], &ok), a1 = fabsf(f64::to_f(wr[2], &ok)),
                        a2 = fabsf(f64::to_f(wr[3], &ok));
            ok = ok && far_from_ties(d0, d1, d2, a1, a2, 0x1p-18f, 0x1p-40f, mp, mp.tie_tol_f);
        }
        if (ok) return false;
    }
    if (mp.scheme != NPW_RBF_ENO_ && mp.scheme != NPW_RBF_WENO_) return false;
    if constexpr (K2) {
        const double w[6] = {0.0, (double)wr[1], (double)wr[2], (double)wr[3], (double)wr[4], 0.0};
        return face_near_tie_k2(w, mp, tol);
    }
    return face_near_tie_d((double)wr[1], (double)wr[2], (double)wr[3], (double)wr[4], mp, tol);
}

// ---------------------------------------------------------------------------------------
// Physical fluxes and wave speeds (Sec. 5.2 examples).  dir 0 = x, 1 = y.
// ---------------------------------------------------------------------------------------
template <typename R, int KIND>
__device__ __forceinline__ void phys_flux(const R* U, const MethodParams& mp, int dir, R* F) {
    if (KIND == NPW_FLUX_ADVECTION_) {
        F[0] = (dir == 0 ? mp_val<R>(mp.adv_speed, mp.adv_speed_f) : mp_val<R>(mp.adv_speed_y, mp.adv_speed_y_f)) * U[0];
    } else if (KIND == NPW_FLUX_BURGERS_) {
        F[0] = R(0.5) * U[0] * U[0];
    } else if (KIND == NPW_FLUX_EULER1D_) {
        const R g = mp_val<R>(mp.gamma, mp.gamma_f);
        R rho = U[0], u = quotient(U[1], rho), E = U[2];
        R P = (g - R(1.0)) * (E - R(0.5) * rho * u * u);
        F[0] = rho * u;
        F[1] = rho * u * u + P;
        F[2] = (E + P) * u;
    } else {
        const R g = mp_val<R>(mp.gamma, mp.gamma_f);
        R rho = U[0], u = quotient(U[1], rho), v = quotient(U[2], rho), E = U[3];
        R P = (g - R(1.0)) * (E - R(0.5) * rho * (u * u + v * v));
        R un = (dir == 0) ? u : v;
        F[0] = rho * un;
        F[1] = U[1] * un + ((dir == 0) ? P : R(0.0));
        F[2] = U[2] * un + ((dir == 0) ? R(0.0) : P);
        F[3] = (E + P) * un;
    }
}

template <typename R, int KIND>
__device__ __forceinline__ R wave_speed(const R* U, const MethodParams& mp, int dir) {
    if (KIND == NPW_FLUX_ADVECTION_)
        return fabs(dir == 0 ? mp_val<R>(mp.adv_speed, mp.adv_speed_f) : mp_val<R>(mp.adv_speed_y, mp.adv_speed_y_f));
    if (KIND == NPW_FLUX_BURGERS_) return fabs(U[0]);
    const R g = mp_val<R>(mp.gamma, mp.gamma_f);
    if (KIND == NPW_FLUX_EULER1D_) {
        R rho = U[0], u = U[1] / rho;
        R P = (g - R(1.0)) * (U[2] - R(0.5) * rho * u * u);
        return fabs(u) + sqrt(g * P / rho);
    }
    R rho = U[0], u = U[1] / rho, v = U[2] / rho;
    R P = (g - R(1.0)) * (U[3] - R(0.5) * rho * (u * u + v * v));
    return fabs(dir == 0 ? u : v) + sqrt(g * P / rho);
}

template <int KIND>
__host__ __device__ constexpr int kind_m() {
    return KIND == NPW_FLUX_EULER1D_ ? 3 : (KIND == NPW_FLUX_EULER2D_ ? 4 : 1);
}

// Lax-Friedrichs flux of one face, all M fields: h = 0.5 (f(a) + f(b) - alpha (b - a)).
template <typename R, int KIND, int M>
__device__ __forceinline__ void lf_flux(const R* a, const R* b, R alpha, const MethodParams& mp, int dir, R* h) {
    R fa[M], fb[M];
    phys_flux<R, KIND>(a, mp, dir, fa);
    phys_flux<R, KIND>(b, mp, dir, fb);
#pragma unroll
    for (int k = 0; k < M; ++k) h[k] = R(0.5) * (fa[k] + fb[k] - alpha * (b[k] - a[k]));
}

// ---------------------------------------------------------------------------------------
// Characteristic variant (1D Euler): Roe average of the two cells at the face, right
// eigenvectors R (columns) of dF/dU and their inverse in closed form,
//   L = [ (b2 + u/c)/2, -(b1 u + 1/c)/2, b1/2 ;  1 - b2, b1 u, -b1 ;  (b2 - u/c)/2, -(b1 u - 1/c)/2, b1/2 ]
// with b1 = (gamma - 1)/c^2, b2 = b1 u^2 / 2.
// ---------------------------------------------------------------------------------------
template <typename R>
__device__ __forceinline__ bool euler_eig(const R* UL, const R* UR, R gamma, R Rm[3][3], R Lm[3][3]) {
    R rl = UL[0], rr = UR[0];
    R ul = UL[1] / rl, ur = UR[1] / rr;
    R pl = (gamma - R(1.0)) * (UL[2] - R(0.5) * rl * ul * ul);
    R pr = (gamma - R(1.0)) * (UR[2] - R(0.5) * rr * ur * ur);
    R hl = (UL[2] + pl) / rl, hr = (UR[2] + pr) / rr;
    R sl = sqrt(rl), sr = sqrt(rr);
    R u = (sl * ul + sr * ur) / (sl + sr);
    R h = (sl * hl + sr * hr) / (sl + sr);
    R c2 = (gamma - R(1.0)) * (h - R(0.5) * u * u);
    if (!(c2 > R(0.0))) return false;
    R c = sqrt(c2);
    Rm[0][0] = R(1.0);
    Rm[0][1] = R(1.0);
    Rm[0][2] = R(1.0);
    Rm[1][0] = u - c;
    Rm[1][1] = u;
    Rm[1][2] = u + c;
    Rm[2][0] = h - u * c;
    Rm[2][1] = R(0.5) * u * u;
    Rm[2][2] = h + u * c;
    R b1 = (gamma - R(1.0)) / c2;
    R b2 = R(0.5) * b1 * u * u;
    R uc = u / c, ic = R(1.0) / c;
    Lm[0][0] = R(0.5) * (b2 + uc);
    Lm[0][1] = R(-0.5) * (b1 * u + ic);
    Lm[0][2] = R(0.5) * b1;
    Lm[1][0] = R(1.0) - b2;
    Lm[1][1] = b1 * u;
    Lm[1][2] = -b1;
    Lm[2][0] = R(0.5) * (b2 - uc);
    Lm[2][1] = R(-0.5) * (b1 * u - ic);
    Lm[2][2] = R(0.5) * b1;
    return true;
}

}  // namespace npw
