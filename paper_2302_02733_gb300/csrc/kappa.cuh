// Synchrotron coefficients of kappa-distributed (or Maxwell-Juttner) electrons by quadrature
// over the distribution: the nonthermal models of the paper's Section 2.1, integrated
// numerically as its outlook (Section 4) proposes. This is the accurate path: it makes the
// surrogate's training set, is the reference the surrogate is checked against, and stands in
// for it outside its box.
//
// Definitions, in an isotropic distribution N(g) (g the Lorentz factor, p = sqrt(g^2 - 1)):
//   kappa:  N = n C g p (1 + (g - 1)/(kappa w))^-(kappa+1), w = (kappa - 3) Theta / kappa;
//   j_I, j_Q, j_V = A int N [F, G, (4/3) cot(theta) H / g](X / g^2) dg,
//     A = sqrt(3) e^3 B sin(theta) / (4 pi m c^2), X = nu / ((3/2) nu_B sin(theta)),
//     F = x int_x K_5/3, G = x K_2/3, H = x K_1/3 + int_x K_1/3 (ultrarelativistic kernels);
//   a_S = -(1 / (2 nu^2 m)) int k_S g^2 d/dg (N / g^2) dg for each kernel k_S;
//   r_V = (2 e^2 nu_B cos / (m c nu^2)) g(X_T) int N asinh(p) / (g p) dg,
//   r_Q = (e^2 nu_B^2 sin^2 / (m c nu^3)) f(X_T) int N (2 g - 1/g) dg,
// with the Shcherbakov corrections f, g at X_T as for the thermal fits, and (j_Q, j_V),
// (a_Q, a_V) kept inside the light cone. For Maxwell-Juttner electrons the rotativity averages
// are exactly K0/K2 and K1/K2 + 6 Theta.
//
// Numerics (device). Both integrals run over s = ln p by the trapezoid rule, which converges
// geometrically for these integrands (they are analytic in s and fall off at both ends), on nodes
// s_lo + k h that do not depend on the point: everything that is a function of p alone comes from a
// table, and a node costs one logarithm and exponential for the distribution and one exponential
// for the kernels. F, G and H come from one piecewise polynomial each of K(x) e^x x^(-1/3) in ln x
// (degree 7 on intervals of 1/8, about 1e-15), built once per context from the trapezoid rule on their
// cosh-integral representations. Two grades:
//  - tabulated (kExact false; the FP32 render, the surrogate's training set and fallback,
//    rt_kappa_coeffs): h = 0.15 (finer above kappa = 10), within about 4e-10 of the integrals;
//  - exact (kExact true; the FP64 render): h = 0.1, about 1e-15;
//  - Maxwell-Juttner electrons (kappa <= 0) at h = 0.025 in both: far above nu_c their integrand is a
//    peak about 0.1 wide.
// It is bound by the FP64 pipe, at about 100 instructions a node that emits and 50 one that does not.
// 8-point Gauss-Legendre panels (16 nodes per unit of s tabulated, 64 exact) with kernels from an
// interpolated table of logarithms (1.6e-8), or in the exact grade summed at every node, took 51.7 ms
// for 60,000 points (now 5.7 to 6.0) and 1.1 to 1.6 s for a 64^2 image (now 14 ms of transfer, with its
// points spread over all lanes), and 58 s for a 20^2 FP64 image (now 11 ms of transfer).
#pragma once
#include "rt_common.cuh"

namespace prt {

// KappaTables (rt_common.cuh): the kernels' polynomials [kSynN][3][8] in ln x from ln 1e-12, interval
// 1/8, and the nodes' functions of p [kKapN][8] at s = ln 1e-4 + 0.025 k.
constexpr double kSynLo = -27.631021115928547;  // ln 1e-12
constexpr int kSynN = 274;                      // up to ln 740 = 6.6067
constexpr double kKapLo = -9.210340371976182;   // ln 1e-4
constexpr double kKapH = 0.025;
constexpr int kKapN = 2000;                     // up to s = 40.8; nodes below and beyond are computed in place

// e^x times F, G, H at x by the trapezoid rule on int_0^inf e^{-x (cosh t - 1)} c(t) dt with
// c = cosh(5t/3)/cosh t, cosh(2t/3), cosh(t/3) and cosh(t/3)/cosh t, at step 0.125 min(1, x^-1/2)
// (the integrand's peak at t = 0 is x^-1/2 wide; the rule converges geometrically for these
// analytic integrands), every cosh from u = e^{t/3}.
__device__ __forceinline__ void synch_kernels_scaled(double x, double k[3]) {
    const double h = 0.125 * fmin(1.0, rsqrt(x));
    double a = 0.5, b = 0.5, c = 0.5, d = 0.5;  // t = 0, half weight: every c(0) = 1
    for (int i = 1; i < 4096; i++) {
        double u = exp(i * h * (1.0 / 3.0)), iu = 1.0 / u;
        double u2 = u * u, iu2 = iu * iu, u3 = u2 * u, iu3 = iu2 * iu;
        double ch = 0.5 * (u3 + iu3), sh = 0.5 * expm1(i * h);  // cosh t - 1 = 2 sinh^2(t/2) = (e^t - 1)^2 / (2 e^t)
        double arg = x * 2.0 * sh * sh * iu3;
        if (arg > 745.0) break;
        double e = exp(-arg), ich = 1.0 / ch;
        double c13 = 0.5 * (u + iu);
        double ta = e * 0.5 * (u3 * u2 + iu3 * iu2) * ich;
        a += ta;
        b += e * 0.5 * (u2 + iu2);
        c += e * c13;
        d += e * c13 * ich;
        if (i > 4 && ta < 1e-19 * a) break;
    }
    k[0] = x * h * a;
    k[1] = x * h * b;
    k[2] = x * h * c + h * d;
}

// The functions of p a node needs: g - 1, p^3 (N dg / q), those of the two rotativity averages,
// 1 / g^2, 2 ln g, 1 / g, p / g (with q the distribution's factor and dg = (p^2 / g) ds).
struct KapNode {
    double gm1, p3, wv, wq, ig2, lg2, ig, pg;
};
__device__ __forceinline__ KapNode kap_node(double s) {
    const double p = exp(s), g = sqrt(1.0 + p * p), ig = 1.0 / g;
    return KapNode{p * p / (g + 1.0), p * p * p, p * p * asinh(p) * ig, p * p * p * (2.0 * g - ig), ig * ig, 2.0 * log(g),
                   ig,  p * ig};
}

__device__ __forceinline__ double shcherbakov_f(double X) {
    double f = 2.011 * exp(-pow(X, 1.035) / 4.7) - cos(0.5 * X) * exp(-pow(X, 1.2) / 2.73) - 0.011 * exp(-X / 47.2);
    if (X > 1.0)
        f += (0.011 * exp(-X / 47.2) - 369.6934286909082 * pow(X, -8.0 / 3.0))  // 2^-1/3 3^-23/6 1e4 pi
             * 0.5 *
             (1.0 + tanh(10.0 * log(X / 120.0)));
    return f;
}

// out: jI jQ jV aI aQ aV rQ rV (cgs). kappa <= 0 selects Maxwell-Juttner electrons. kExact:
// the exact grade, else the tabulated one.
template <bool kExact = false>
__device__ __forceinline__ void kappa_coeffs_quad(const KappaTables &T, double ne, double Te, double B, double nu,
                                                  double thB, double kappa, double out[8]) {
#pragma unroll
    for (int i = 0; i < 8; i++) out[i] = 0.0;
    if (!(ne > 0.0) || !(Te > 0.0) || !(B > 0.0) || !(nu > 0.0)) return;
    if (kappa > 0.0 && !(kappa > 3.0)) return;
    const bool thermal = kappa <= 0.0;
    const double Td = fmax(Te, 1e-60);  // the distribution's: below, powers of p leave the FP64 range
    const double kw = thermal ? 1.0 : (kappa - 3.0) * Td, ikw = 1.0 / kw, kp1 = kappa + 1.0;
    const double ite = 1.0 / Td, s0 = thermal ? ite : kp1 * ikw;  // s0: -(dln q/dg) at g = 1
    double s_hi;
    if (thermal) {
        const double ghi1 = 800.0 * Td;
        s_hi = 0.5 * log(ghi1 * (ghi1 + 2.0));
    } else {
        s_hi = log((1.0 + kw) * 10.0) + fmin(45.0 / (kappa - 2.34), 600.0);
    }
    // hotter: p^3 leaves the FP64 range on the way to s_hi (and an infinite s_hi, of an infinite Theta_e or
    // kappa, would be 2^31 nodes)
    if (!(s_hi < 236.0)) return;
    // the step by the distribution's steepness (toward large kappa it narrows to the Maxwell-Juttner
    // one). Worst errors over Theta_e 0.1 to 10 and X to 3e5: tabulated 4e-10 below kappa = 10, 7e-13,
    // 4e-14 and 2e-15 in the others, exact 9e-16, 9e-13 (where j is 1e-30 of its scale) and 4e-15.
    // At X = 10, where the range's lower end counts: tabulated 2e-12 (kappa = 3.001: 3e-10), exact
    // 7e-13 (7e-12)
    const int stride = thermal ? 1
                       : kExact ? (kappa < 3.1 ? 1 : kappa < 10.0 ? 4 : kappa < 20.0 ? 3 : kappa < 99.0 ? 2 : 1)
                                : (kappa < 10.0 ? 6 : kappa < 20.0 ? 4 : kappa < 40.0 ? 3 : 1);
    const double h = stride * kKapH;
    const double s = sin(thB), c = cos(thB), as = fabs(s);
    const double nuB = kQe * B / (2.0 * kPi * kMe * kC);
    const bool emits = !(as < 1e-12);
    const double X = emits ? nu / (1.5 * nuB * as) : 0.0, lX = emits ? log(X) : 0.0;
    // the integrals in units of h. The first node stands for the range below it too: the integrands
    // go as p^c there, c = 3 (those of dN/dg as p, p^3 and p^5), and a sum h f_0 / (1 - e^-ch) from
    // -infinity less the integral f_0 / c below s_lo leaves h f_0 w_c. The momenta of cold electrons (p
    // of sqrt(2 / s0) and above) come down to s_lo: their nodes begin at s0 p^2 = 2e-6, whatever that
    // is, and nothing is left out below
    const bool cold = s0 > 5e4;
    const int k0 = cold ? (int)floor((0.5 * log(2e-6 / s0) - kKapLo) / h) : 0;
    const double w1 = 1.0 / (1.0 - exp(-h)) - (cold ? 0.0 : 1.0 / h),
                 w3 = 1.0 / (1.0 - exp(-3.0 * h)) - (cold ? 0.0 : 1.0 / (3.0 * h)),
                 w5 = 1.0 / (1.0 - exp(-5.0 * h)) - (cold ? 0.0 : 1.0 / (5.0 * h));
    double nacc = 0.0, rv = 0.0, rq = 0.0, e[6] = {0, 0, 0, 0, 0, 0}, fq = 0.0;
    // for g >> kappa w all integrands are powers of p (to 1e-16 from here), and the tail has a closed form
    const double s_pow = thermal ? s_hi : 37.0 + log(1.0 + kw);
    const int K = (int)floor((fmin(s_hi, s_pow) - kKapLo) / h + 1e-9);
    bool on = emits;
    for (int k = k0; k <= K; k++) {
        const int ik = k * stride;
        const KapNode n = (unsigned)ik < (unsigned)kKapN ? T.node[ik] : kap_node(kKapLo + ik * kKapH);
        double q, slope;  // N / n up to its norm is g p q; -(dln q/dg)
        const double kg = kw + n.gm1;
        if (thermal) {
            q = exp(-n.gm1 * ite);
            slope = ite;
        } else {
            // the rounding of the quotient kg / kw is raised to the power kappa: 1e-10 of q at kappa = 1e6.
            // Below 10 that is as small as log1p's own, and 60,000 points of kappa 3 to 8 take 6.16 ms
            // against 6.22 (points of kappa 1e5, 21.4 ms against 22.0 with the quotient's logarithm)
            q = exp(-kp1 * (kappa < 10.0 ? log(kg * ikw) : log1p(n.gm1 * ikw)));
            slope = 0.0;
        }
        const double f3 = k == k0 ? w3 : 1.0;
        const double N = n.p3 * q * f3;
        nacc += N;
        rv += n.wv * q * f3;
        fq = n.wq * q;
        rq += fq * f3;
        const double x = X * n.ig2;
        if (on && x < 740.0) {
            if (!thermal) slope = kp1 / kg;
            double D = (n.pg - n.p3 * slope) * q;
            if (k == k0) {  // p, p^3 and p^5 apart: q = 1 - s0 (g - 1) + .., slope q = s0 (1 + ..)
                const double d1 = -s0 * n.gm1;
                D = n.pg * (w1 + d1 * w3 + ((q - 1.0) - d1) * w5) - n.p3 * s0 * (w3 + (slope * q / s0 - 1.0) * w5);
            }
            const double lx = lX - n.lg2, v = (lx - kSynLo) * 8.0;
            const double E = exp(lx * (1.0 / 3.0) - x);
            int i = v > 0.0 ? (int)v : 0;
            i = i < kSynN - 1 ? i : kSynN - 1;
            // below the table (x < 1e-12) F and G go as x^(1/3) and H is constant
            const double t = v > 0.0 ? 2.0 * (v - i) - 1.0 : -1.0;
            const double EH = v > 0.0 ? E : exp(kSynLo * (1.0 / 3.0) - x);
            const double *P = T.kern + 24 * i;
            double K0 = P[7], K1 = P[15], K2 = P[23];
#pragma unroll
            for (int m = 6; m >= 0; m--) {
                K0 = fma(K0, t, P[m]);
                K1 = fma(K1, t, P[8 + m]);
                K2 = fma(K2, t, P[16 + m]);
            }
            K0 *= E;
            K1 *= E;
            K2 *= EH * n.ig;
            e[0] += N * K0;
            e[1] += N * K1;
            e[2] += N * K2;
            e[3] += D * K0;
            e[4] += D * K1;
            e[5] += D * K2;
            // beyond their peak the emission's terms fall off as powers of p: they end where they are
            // below an eighth of a unit in the last place of each sum. Not above x = 1, where the kernels
            // rise by e^x yet: the terms of cold electrons pass a peak of their own there, which may lie
            // far above what follows it and far below the power-law tail's
            if ((k & 7) == 0 && x < 1.0)
                on = !(N * K0 <= 1e-17 * e[0] && N * K2 <= 1e-17 * e[2] && fabs(D * K0) <= 1e-17 * fabs(e[3]) &&
                       fabs(D * K2) <= 1e-17 * fabs(e[5]) && e[0] > 0.0);
        }
    }
    if (!thermal) {
        // the Faraday-conversion average beyond the last node, up to s_hi, where its integrand is
        // f e^{-c (s - s_K)} with c = kappa - 3: the sum to infinity, less the integral beyond s_hi
        // (the other integrals fall off faster and have nothing left there)
        const double cc = kappa - 3.0, ch = cc * h, d = s_hi - (kKapLo + K * h);
        const double a = ch < 0.05 ? h * (-0.5 + ch * (1.0 / 12.0) - ch * ch * ch * (1.0 / 720.0)) : h / expm1(ch) - 1.0 / cc;
        rq += fq * (a - expm1(-cc * d) / cc) / h;
    }
    const double inorm = 1.0 / nacc;  // the distribution's normalisation
    rv *= inorm;
    rq *= inorm;
#pragma unroll
    for (int j = 0; j < 6; j++) e[j] *= inorm;
    double Xr = Te * sqrt(1.4142135623730951 * as * 1.0e3 * nuB / nu);
    out[6] = ne * kQe * kQe * nuB * nuB * s * s / (kMe * kC * nu * nu * nu) * shcherbakov_f(Xr) * rq;
    out[7] = 2.0 * ne * kQe * kQe * nuB * c / (kMe * kC * nu * nu) * (1.0 - 0.11 * log1p(0.035 * Xr)) * rv;
    if (!emits) return;
    double A = 1.7320508075688772 * kQe * kQe * kQe * B * as / (4.0 * kPi * kMe * kC * kC);
    double cot = c / s;
    double jI = ne * A * e[0], jQ = ne * A * e[1], jV = ne * A * (4.0 / 3.0) * cot * e[2];
    double ab = -ne * A / (2.0 * nu * nu * kMe);
    double aI = ab * e[3], aQ = ab * e[4], aV = ab * (4.0 / 3.0) * cot * e[5];
    if (!(jI > 1e-250)) return;
    double pj = sqrt((jQ / jI) * (jQ / jI) + (jV / jI) * (jV / jI));
    if (pj > 1.0) {
        jQ /= pj;
        jV /= pj;
    }
    if (aI > 0.0) {
        double pa = sqrt((aQ / aI) * (aQ / aI) + (aV / aI) * (aV / aI));
        if (pa > 1.0) {
            aQ /= pa;
            aV /= pa;
        }
    }
    out[0] = jI;
    out[1] = jQ;
    out[2] = jV;
    out[3] = aI;
    out[4] = aQ;
    out[5] = aV;
}

}  // namespace prt
