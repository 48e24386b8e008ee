// FP64 tables of functions of one positive variable, for the thermal rotativities: a polynomial on each
// sixteenth (or sixty-fourth) of an octave, found from the exponent and the top mantissa bits, in the
// rest of the mantissa (as u = -1/2 .. 1/2, one FP64 instruction). Two functions to a segment, D + 1
// coefficients each, D + 1 Chebyshev nodes behind them.
#pragma once

namespace prt {

// The segment of v >= 2^e0 (2^bits segments an octave) and its variable u; negative below 2^e0.
__device__ __forceinline__ int therm_segment(double v, int bits, int e0, double &u) {
    const long long b = __double_as_longlong(v);
    u = __longlong_as_double(((long long)((unsigned long long)b << bits) & 0x000fffffffffffffll) | 0x3ff0000000000000ll) - 1.5;
    return (int)(b >> (52 - bits)) - ((1023 + e0) << bits);
}
template <int D>
__device__ __forceinline__ void therm_eval(const double *t, double u, double &a, double &b) {
    a = t[D];
    b = t[2 * D + 1];
#pragma unroll
    for (int k = D - 1; k >= 0; k--) {
        a = fma(a, u, t[k]);
        b = fma(b, u, t[D + 1 + k]);
    }
}

//  - bes: K0/K2 and K1/K2 of z = 1/Theta for Theta from 2^-40 (1e-12) to 2^20;
//  - shc: Shcherbakov's f(X) and 1 - 0.11 ln(1 + 0.035 X) for X from 2^-30 to 2^14.
// A fit converges as rho^-(D + 1), with rho from the distance to the function's nearest singular point in
// halves of a segment. The Bessel ratios and the logarithm have none nearer than 32 of them (rho 64).
// f's switch 1 - 1/((X/120)^20 + 1) has poles at 120 exp(+-i pi/20), 18.8 off the real line: with 16
// segments an octave rho is 19 below X = 128 and 12 from there, which left 1.5e-14 and 1.6e-12 of f's
// terms in the octaves beside it; with 64 segments there, 0.8e-15, as evaluated directly. From 256 on they
// are far enough (1.1e-15).
// 17 and 19 FP64 instructions in place of 27 reciprocal square roots (14 series terms at z < 2) and of
// 11 transcendental functions; the FP64 pipe bounds the kernels that read them. With fmks_y64 the FP64
// instructions of 32 states went from 1,721 to 1,343 and the points of a torus at 200^2 from 51 to 36 ms; an
// ADAF's transfer at 64^2 from 16.4 to 9.5 ms.
struct ThermTab {
    static constexpr int db = 8, ds = 9;                                  // degrees
    static constexpr int eb = -40, nb = 60 * 16, es = -30, ns = 44 * 16;  // first octave, segments
    static constexpr int ef = 6, nf = 2 * 64;                             // finer ones for f: octaves 64 and 128
    static constexpr int bes = 0, shc = nb * 2 * (db + 1), size = shc + (ns + nf) * 2 * (ds + 1);

    // The segment of shc that holds X and its variable; -1 outside the table.
    static __device__ __forceinline__ int shc_segment(double X, double &u) {
        const bool fine = (unsigned)(__double_as_longlong(X) >> 48) - ((1023u + ef) << 4) < 2u * 16u;
        const int i = therm_segment(X, fine ? 6 : 4, fine ? ef : es, u);
        return fine ? ns + i : ((unsigned)i < (unsigned)ns ? i : -1);
    }
    // Node j of segment i of a table that starts at octave e0, 2^bits segments each; x: the Chebyshev node.
    static __device__ __forceinline__ double at(int i, int bits, int e0, double x) {
        const int n = 1 << bits;
        return ldexp(1.0 + ((i & (n - 1)) + 0.5 + 0.5 * x) / n, e0 + (i >> bits));
    }
};

// Chebyshev coefficient k of the polynomial through f at the nodes x_j = cos(pi (j + 1/2) / (D + 1)), and from
// all of them the coefficients in u.
template <int D>
__device__ __forceinline__ double therm_chebyshev(const double f[D + 1], int k) {
    double s = 0.0;
    for (int q = 0; q <= D; q++) s += f[q] * cospi(k * (q + 0.5) / (D + 1));
    return s * (k == 0 ? 1.0 : 2.0) / (D + 1);
}
template <int D>
__device__ __forceinline__ void therm_powers(const double ch[D + 1], double p[D + 1]) {
    double a[D + 1], b[D + 1];  // T_k and T_k+1 in powers of x = 2 u
    for (int q = 0; q <= D; q++) p[q] = 0.0, a[q] = q == 0, b[q] = q == 1;
    for (int k = 0; k <= D; k++) {
        double c[D + 1];
        for (int q = 0; q <= D; q++) {
            p[q] += ch[k] * a[q];
            c[q] = (q > 0 ? 2.0 * b[q - 1] : 0.0) - a[q];
        }
        for (int q = 0; q <= D; q++) a[q] = b[q], b[q] = c[q];
    }
    for (int q = 0; q <= D; q++) p[q] = ldexp(p[q], q);
}

}  // namespace prt
