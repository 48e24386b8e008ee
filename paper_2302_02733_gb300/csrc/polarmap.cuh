// The polar map of the FMKS grid in FP64: mu = theta - pi/2 as a function of y = X2 - 1/2 at blend weight
// w, and its inverse. fmks_mu of transfer.cuh is the FP32 transfer's and the table's.
// kPi, kX2TabW and kX2TabT come from rt_common.cuh, which its includer has.
#pragma once

namespace prt {

// mu, d theta / d X2 and theta_j - theta_g at y.
template <class Grid>
__device__ __forceinline__ double fmks_map64(const Grid &g, double w, double y, double &dth2, double &dd) {
    double s, c;
    sincospi(2.0 * y, &s, &c);
    const double omh = 1.0 - g.hslope, ya = pow(fabs(2.0 * y / g.poly_xt), g.poly_alpha);
    const double g0 = kPi * y - 0.5 * omh * s, g1 = kPi - kPi * omh * c;
    dd = 2.0 * g.poly_norm * y * (1.0 + ya / (g.poly_alpha + 1.0)) - g0;
    dth2 = fma(w, 2.0 * g.poly_norm * (1.0 + ya) - g1, g1);
    return fma(w, dd, g0);
}

// y = X2 - 1/2 of the point at polar angle th (mu = th - pi/2) in FP64, with one evaluation of the map: at the table's guess (within 1.3e-5 of the root) the
// four derivatives of mu follow from the values already there, so one fourth-order step reaches the
// root (the error is the step's fourth power, 3e-20, times the map's fourth derivative), and d theta /
// d X2 and theta_j - theta_g are carried from the guess to the root by their Taylor series. Two Newton
// steps and the values at the root took three evaluations of the map, each a sine, cosine and power.
// A guess further off (a coarse spot of the table) takes Newton's steps, kept within the bracket that
// they leave.
template <class Grid>
__device__ __forceinline__ double fmks_y64(const Grid &g, double w, double th, double mu, double &dth2, double &dd) {
    const double fw = w * (kX2TabW - 1), ft = th * ((kX2TabT - 1) / kPi);
    const int iw = min(max((int)fw, 0), kX2TabW - 2), it = min(max((int)ft, 0), kX2TabT - 2);
    const double tw = fw - iw, tt = ft - it;
    const double *T = g.x2_table + iw * kX2TabT + it;
    const double y0 = (1.0 - tw) * ((1.0 - tt) * T[0] + tt * T[1]) + tw * ((1.0 - tt) * T[kX2TabT] + tt * T[kX2TabT + 1]) - 0.5;
    double s, c;
    sincospi(2.0 * y0, &s, &c);
    const double omh = 1.0 - g.hslope, N = g.poly_norm, al = g.poly_alpha, ay = fabs(y0);
    const double ya = ay > 0.0 ? exp(al * log(2.0 * ay / g.poly_xt)) : 0.0;
    const double iy = ay > 1e-100 ? 1.0 / y0 : 0.0;
    // theta_g - pi/2 and theta_j - theta_g with four derivatives each
    const double tp = 2.0 * kPi, g0 = kPi * y0 - 0.5 * omh * s, g1 = kPi - kPi * omh * c, g2 = kPi * tp * omh * s,
                 g3 = tp * tp * kPi * omh * c, g4 = -tp * tp * g2;
    const double j2 = 2.0 * N * ya * al * iy, j3 = j2 * (al - 1.0) * iy, j4 = j3 * (al - 2.0) * iy;
    const double d0 = 2.0 * N * y0 * (1.0 + ya / (al + 1.0)) - g0, d1 = 2.0 * N * (1.0 + ya) - g1, d2 = j2 - g2, d3 = j3 - g3,
                 d4 = j4 - g4;
    const double f1 = fma(w, d1, g1), f2 = fma(w, d2, g2), f3 = fma(w, d3, g3), f4 = fma(w, d4, g4), if1 = 1.0 / f1;
    const double x = (mu - fma(w, d0, g0)) * if1, b = 0.5 * f2 * if1, e = f3 * if1 * (1.0 / 6.0);
    double y = y0 + x * (1.0 + x * (-b + x * (2.0 * b * b - e)));
    // what the step leaves out is x^4 (f4 / 24 f1 + 5 b^3), what dd's series does x^4 d4 / 24; below alpha
    // = 4 the map's higher derivatives are singular at y = 0 (at alpha = 1 the second one jumps there,
    // unseen by f4)
    const double xx = x * x;
    if (!(fabs(x) < 3e-5 && fabs(b * x) < 1e-4 && xx * xx * (fabs(f4) + fabs(d4)) <= 2e-15 * f1 && (al >= 4.0 || fabs(x) < ay))) {
        double lo = -0.5, hi = 0.5;
        y = y0;
        for (int k = 0; k < 80; k++) {
            const double f = fmks_map64(g, w, y, dth2, dd) - mu, yn = y - f / dth2;
            if (fabs(yn - y) <= 1e-16) break;
            (f < 0.0 ? lo : hi) = y;
            y = yn > lo && yn < hi ? yn : 0.5 * (lo + hi);
        }
        return y;
    }
    y = fmin(fmax(y, -0.5), 0.5);
    const double t = y - y0;
    dth2 = fma(t, fma(0.5 * t, fma(t * (1.0 / 3.0), f4, f3), f2), f1);
    dd = fma(t, fma(0.5 * t, fma(t * (1.0 / 3.0), d3, d2), d1), d0);
    return y;
}

}  // namespace prt
