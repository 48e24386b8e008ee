// The polar map of the FMKS grid, mu = theta - pi/2 as a function of y = X2 - 1/2 at blend weight w =
// exp(s (X1_in - X1)), and its inverse. With x2 = 1/2 + y, sin(2 pi x2) = -sin(2 pi y) and cos(2 pi x2) =
// -cos(2 pi y), so every term is small near the equator and an FP32 evaluation keeps the relative precision
// of mu there. kPi, kX2TabW and kX2TabT come from rt_common.cuh and the small integers' conversions from
// ffloat.cuh, which its includer has.
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

// The map and its inverse in FP32, by the same one evaluation and step. Every sum and product is rounded
// by itself (no contraction is left to the compiler), so that all kernels that this is inlined into get
// the same bits, from the table's guess on.
template <class Grid>
__device__ __forceinline__ float fmks_map32(const Grid &g, float w, float y, float &dth2, float &dd) {
    float s, c;
    sincospif(__fmul_rn(2.0f, y), &s, &c);
    const float omh = __fadd_rn(1.0f, -g.f_hslope), pi = (float)kPi, yp = __fmul_rn(2.0f, y);
    const float ya = powf(fabsf(__fdiv_rn(yp, g.f_poly_xt)), g.f_poly_alpha);
    const float g0 = __fmaf_rn(pi, y, __fmul_rn(__fmul_rn(-0.5f, omh), s)), g1 = __fmul_rn(pi, __fmaf_rn(-omh, c, 1.0f));
    const float np = __fmul_rn(g.f_poly_norm, yp), n2 = __fmul_rn(2.0f, g.f_poly_norm);
    dd = __fadd_rn(__fmaf_rn(np, __fdividef(ya, g.f_poly_alpha1), np), -g0);
    dth2 = __fmaf_rn(w, __fadd_rn(__fmaf_rn(n2, ya, n2), -g1), g1);
    return __fmaf_rn(w, dd, g0);
}

// A torus at 1024^2: points and chain 57.7 -> 53.6 ms, the unpolarized transfer 34.8 -> 30.0 (three
// evaluations of the map in one).
template <class Grid>
__device__ __forceinline__ float fmks_y32(const Grid &g, float w, float th, float mu, float &dth2, float &dd) {
    const float fw = __fmul_rn(w, float(kX2TabW - 1)), ft = __fmul_rn(th, float((kX2TabT - 1) / kPi));
    // fw in [0, 63], ft in [0, 1023]: no conversion instructions
    const int iw = min(max(floor_small(fw), 0), kX2TabW - 2), it = min(max(floor_small(ft), 0), kX2TabT - 2);
    const float tw = __fadd_rn(fw, -i2f_small(iw)), tt = __fadd_rn(ft, -i2f_small(it));
    const float *T = g.x2_table_f + iw * kX2TabT + it;
    const float a0 = __fmaf_rn(tt, __fadd_rn(T[1], -T[0]), T[0]),
                a1 = __fmaf_rn(tt, __fadd_rn(T[kX2TabT + 1], -T[kX2TabT]), T[kX2TabT]);
    const float y0 = __fadd_rn(__fmaf_rn(tw, __fadd_rn(a1, -a0), a0), -0.5f);
    float s, c;
    sincospif(__fmul_rn(2.0f, y0), &s, &c);
    const float omh = __fadd_rn(1.0f, -g.f_hslope), pi = (float)kPi, yp = __fmul_rn(2.0f, y0), al = g.f_poly_alpha;
    const float ay = fabsf(y0), ya = powf(fabsf(__fdiv_rn(yp, g.f_poly_xt)), al);
    const float iy = ay > 1e-30f ? __fdividef(1.0f, y0) : 0.0f;
    const float po = __fmul_rn(pi, omh), tp = (float)(2.0 * kPi), tp2 = (float)(4.0 * kPi * kPi);
    const float np = __fmul_rn(g.f_poly_norm, yp), n2 = __fmul_rn(2.0f, g.f_poly_norm);
    const float g0 = __fmaf_rn(pi, y0, __fmul_rn(__fmul_rn(-0.5f, omh), s)), g1 = __fmul_rn(pi, __fmaf_rn(-omh, c, 1.0f)),
                g2 = __fmul_rn(__fmul_rn(tp, po), s), g3 = __fmul_rn(__fmul_rn(tp2, po), c), g4 = __fmul_rn(-tp2, g2);
    const float j2 = __fmul_rn(__fmul_rn(__fmul_rn(n2, ya), al), iy), j3 = __fmul_rn(__fmul_rn(j2, __fadd_rn(al, -1.0f)), iy),
                j4 = __fmul_rn(__fmul_rn(j3, __fadd_rn(al, -2.0f)), iy);
    const float d0 = __fadd_rn(__fmaf_rn(np, __fdividef(ya, g.f_poly_alpha1), np), -g0),
                d1 = __fadd_rn(__fmaf_rn(n2, ya, n2), -g1), d2 = __fadd_rn(j2, -g2), d3 = __fadd_rn(j3, -g3), d4 = __fadd_rn(j4, -g4);
    const float f1 = __fmaf_rn(w, d1, g1), f2 = __fmaf_rn(w, d2, g2), f3 = __fmaf_rn(w, d3, g3), f4 = __fmaf_rn(w, d4, g4);
    const float if1 = __fdividef(1.0f, f1), x = __fmul_rn(__fadd_rn(mu, -__fmaf_rn(w, d0, g0)), if1);
    const float b = __fmul_rn(__fmul_rn(0.5f, f2), if1), e = __fmul_rn(__fmul_rn(f3, if1), 1.0f / 6.0f), xx = __fmul_rn(x, x);
    float y = __fmaf_rn(x, __fmaf_rn(x, __fmaf_rn(x, __fmaf_rn(__fmul_rn(2.0f, b), b, -e), -b), 1.0f), y0);
    if (!(fabsf(x) < 1e-3f && fabsf(__fmul_rn(b, x)) < 2e-3f &&
          __fmul_rn(__fmul_rn(xx, xx), __fadd_rn(fabsf(f4), fabsf(d4))) <= __fmul_rn(1e-8f, f1) && (al >= 4.0f || fabsf(x) < ay))) {
        float lo = -0.5f, hi = 0.5f;
        y = y0;
        for (int k = 0; k < 40; k++) {
            const float f = __fadd_rn(fmks_map32(g, w, y, dth2, dd), -mu), yn = __fmaf_rn(-f, __fdividef(1.0f, dth2), y);
            if (fabsf(__fadd_rn(yn, -y)) <= 3e-8f) break;
            (f < 0.0f ? lo : hi) = y;
            y = yn > lo && yn < hi ? yn : __fmul_rn(0.5f, __fadd_rn(lo, hi));
        }
        return y;
    }
    y = fminf(fmaxf(y, -0.5f), 0.5f);
    const float t = __fadd_rn(y, -y0), t3 = __fmul_rn(t, 1.0f / 3.0f), th2 = __fmul_rn(0.5f, t);
    dth2 = __fmaf_rn(t, __fmaf_rn(th2, __fmaf_rn(t3, f4, f3), f2), f1);
    dd = __fmaf_rn(t, __fmaf_rn(th2, __fmaf_rn(t3, d3, d2), d1), d0);
    return y;
}

}  // namespace prt
