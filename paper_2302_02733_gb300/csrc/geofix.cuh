// The geodesic's RK4 step in 64-bit fixed point on the integer pipes.
//
// GB300 issues 1.6 FP64 thread operations per clock and SM (measured: one FP64 warp instruction per
// 80 clocks and SM sub-partition), but 24 32x32->64-bit multiply-adds and 50 to 90 other 32-bit
// integer operations. A 64-bit fixed-point product and sum take 15 to 18 clocks, so the step runs
// several times faster here than on the FP64 pipe, and carries more bits: the null momentum's
// components share one scale, which bounds every term, so no product or sum needs an exponent of
// its own. Against the same step in extended precision the new r, theta and phi are 30% closer than
// the FP64 form's and the momentum as close (its FP64 rounding dominates); whole rays end 20 to 30%
// closer to those traced in quadruple precision.
//
// Scaling, once per step. rho = 2^e with r / rho in [1/2, 1); x = r / rho, alpha = a / rho. The
// momentum is taken as W, R = K^r, v = rho K^theta and u = rho sin(theta) K^phi, divided by a
// 2^kap that puts the largest below 1/4 (the physical components of a null vector, so all are
// bounded by the same number). Far from the hole v, u and the spin are small beside W and R, and
// an absolute error in v or u moves the ray's impact parameter by r times that: so they are kept 2^g
// times larger (g <= e - 1, which keeps |alpha| 2^g below 1/2). K^phi alone grows as 1 / sin(theta) toward the axis: P = rho K^phi 2^-kap
// 2^-z, u = s P 2^z (P, v and u times 2^g). The affine step becomes hh = h 2^kap / rho, and every rate is dimensionless.
//
// Fx<Q> is a signed 64-bit integer m standing for m 2^-Q. A product of Fx<A> and Fx<B> is
// Fx<A + B - 64>; sums need equal Q. The bound of each quantity is written beside it, with
// |W|, |R|, |v|, |u|, |P| <= 5/16 and 0.45 <= x <= 1.1 through the step's stages. A step that
// leaves these bounds at a stage, starts inside r = 1 or comes near the axis (sin < 2^-10, or a
// polar passage at c u^2 / s >= 1) is taken by the FP64 form instead (fx_step returns false).
#pragma once
#include "ffloat.cuh"

namespace prt {

typedef long long fx64;

__device__ __forceinline__ fx64 fx_shl(fx64 m, int n) { return (fx64)((unsigned long long)m << n); }
// A 64-bit value as signed halves: value = h 2^32 + l.
struct FxHalves {
    int h, l;
};
__device__ __forceinline__ FxHalves fx_halves(fx64 m) {
    const unsigned l = (unsigned)m;
    return FxHalves{(int)((unsigned)((unsigned long long)m >> 32) + (l >> 31)), (int)l};
}
// The high word of a b plus c, and the 64-bit a b + c. Written as single PTX instructions: from
// the same products in C++ the compiler makes 19 instructions of one fixed-point product and its
// sum, from these 7 to 9 (measured: 31 clocks a warp and SM sub-partition against 15 to 18).
__device__ __forceinline__ int fx_madhi(int a, int b, int c) {
#ifdef __CUDA_ARCH__
    int r;
    asm("mad.hi.s32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
#else
    return (int)(((fx64)a * b) >> 32) + c;
#endif
}
__device__ __forceinline__ fx64 fx_madwide(int a, int b, fx64 c) {
#ifdef __CUDA_ARCH__
    fx64 r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return (fx64)a * b + c;
#endif
}
// a b / 2^64 from three of the four partial products (the lowest is below the result's last bit),
// within two units: the middle products' high words are each rounded down, which the constant
// makes up for on average. For |a b| < 2^126.
__device__ __forceinline__ fx64 fx_mulhi(fx64 a, fx64 b) {
    const FxHalves x = fx_halves(a), y = fx_halves(b);
    return fx_madwide(x.h, y.h, (fx64)fx_madhi(x.l, y.h, fx_madhi(x.h, y.l, 1)));
}
// a b / 2^(64 - N), rounded, N = 1 or 2, for |a b| < 2^(126 - N): the same product N bits finer,
// where the rates and a step's last sums would feel the coarser one's unit.
template <int N>
__device__ __forceinline__ fx64 fx_mulfine(fx64 a, fx64 b) {
    const FxHalves x = fx_halves(a), y = fx_halves(b);
    const fx64 m = fx_madwide(x.l, y.h, fx_madwide(x.h, y.l, 1ll << (31 - N)));
    return fx_shl(fx_madwide(x.h, y.h, 0), N) + (m >> (32 - N));
}
// (a b + c d) / 2^63, rounded, for |a b + c d| < 2^125 and middle products below 2^63 in sum
__device__ __forceinline__ fx64 fx_dotfine(fx64 a, fx64 b, fx64 c, fx64 d) {
    const FxHalves x = fx_halves(a), y = fx_halves(b), z = fx_halves(c), w = fx_halves(d);
    const fx64 m = fx_madwide(x.l, y.h, fx_madwide(x.h, y.l, 1ll << 30)) >> 1;
    const fx64 n = fx_madwide(z.l, w.h, fx_madwide(z.h, w.l, 0)) >> 1;
    return fx_shl(fx_madwide(z.h, w.h, fx_madwide(x.h, y.h, 0)), 1) + ((m + n) >> 30);
}
// (a b + c d) / 2^64 with one sign extension for both products; the middle products' high words
// stay below 2^31 in sum for |a|, .. <= 2^62.5.
__device__ __forceinline__ fx64 fx_dothi(fx64 a, fx64 b, fx64 c, fx64 d) {
    const FxHalves x = fx_halves(a), y = fx_halves(b), z = fx_halves(c), w = fx_halves(d);
    const int m = fx_madhi(z.l, w.h, fx_madhi(z.h, w.l, fx_madhi(x.l, y.h, fx_madhi(x.h, y.l, 2))));
    return fx_madwide(z.h, w.h, fx_madwide(x.h, y.h, (fx64)m));
}

#ifndef FX_FITS  // a test's check that a left shift or a sum keeps its value
#define FX_FITS(ok)
#endif

template <int Q>
struct Fx {
    fx64 m;
    template <int N>
    __device__ __forceinline__ Fx<Q + N> up() const {  // the same value, N more fraction bits
        FX_FITS(fx_shl(m, N) >> N == m);
        return Fx<Q + N>{fx_shl(m, N)};
    }
    template <int N>
    __device__ __forceinline__ Fx<Q - N> dn() const {
        return Fx<Q - N>{m >> N};
    }
    __device__ __forceinline__ Fx<Q - 1> twice() const { return Fx<Q - 1>{m}; }  // twice the value
    __device__ __forceinline__ Fx<Q> over(int n) const { return Fx<Q>{m >> n}; }  // value / 2^n
    __device__ __forceinline__ Fx<Q> operator-() const { return Fx<Q>{-m}; }
};
template <int A, int B>
__device__ __forceinline__ Fx<A + B - 64> operator*(Fx<A> a, Fx<B> b) {
    return Fx<A + B - 64>{fx_mulhi(a.m, b.m)};
}
template <int Q>
__device__ __forceinline__ Fx<Q> operator+(Fx<Q> a, Fx<Q> b) {
    FX_FITS(((a.m >> 1) + (b.m >> 1) < (1ll << 62) - 1) && ((a.m >> 1) + (b.m >> 1) > -(1ll << 62)));
    return Fx<Q>{a.m + b.m};
}
template <int Q>
__device__ __forceinline__ Fx<Q> operator-(Fx<Q> a, Fx<Q> b) {
    FX_FITS(((a.m >> 1) - (b.m >> 1) < (1ll << 62) - 1) && ((a.m >> 1) - (b.m >> 1) > -(1ll << 62)));
    return Fx<Q>{a.m - b.m};
}

template <int N, int A, int B>
__device__ __forceinline__ Fx<A + B - 64 + N> fx_fine(Fx<A> a, Fx<B> b) {
    return Fx<A + B - 64 + N>{fx_mulfine<N>(a.m, b.m)};
}
template <int A, int B, int C>
__device__ __forceinline__ Fx<A + B - 63> fx_dot_fine(Fx<A> a, Fx<B> b, Fx<C> c, Fx<A + B - C> d) {
    return Fx<A + B - 63>{fx_dotfine(a.m, b.m, c.m, d.m)};
}
// a b + c d
template <int A, int B, int C>
__device__ __forceinline__ Fx<A + B - 64> fx_dot(Fx<A> a, Fx<B> b, Fx<C> c, Fx<A + B - C> d) {
    return Fx<A + B - 64>{fx_dothi(a.m, b.m, c.m, d.m)};
}

__device__ __forceinline__ int fx_clz(unsigned long long v) {
#ifdef __CUDA_ARCH__
    return __clzll((long long)v);
#else
    return v ? __builtin_clzll(v) : 64;
#endif
}

// d 2^sh as an integer (rounded toward zero): the significand shifted to its place.
__device__ __forceinline__ fx64 fx_from(double d, int sh) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(d);
    const int ex = (int)((b >> 52) & 0x7ffull);
    const unsigned long long s = ((b & 0x000fffffffffffffull) | (ex ? (1ull << 52) : 0ull)) << 10;  // below 2^63
    const int n = 1085 - ex - sh;  // d = s 2^(ex - 1085)
    const fx64 m = n > 63 ? 0 : (fx64)(s >> (n < 0 ? 0 : n));
    return (fx64)b < 0 ? -m : m;
}

// m 2^-sh as a double, rounded to nearest with integer operations (a conversion would take the
// FP64 pipe). For results in the normal range.
__device__ __forceinline__ double fx_to(fx64 m, int sh) {
    if (m == 0) return 0.0;
    const unsigned long long a = m < 0 ? 0ull - (unsigned long long)m : (unsigned long long)m;
    const int z = fx_clz(a);
    const unsigned long long n = a << z;  // top bit set
    unsigned long long q = (n >> 11) + ((n >> 10) & 1ull);
    // exponent field of 2^(63 - z) at the implicit bit's place, added so that a carry of the
    // rounding moves into it
    q += (unsigned long long)(63 - z - sh + 1023 - 1) << 52;
    return __longlong_as_double((long long)(q | ((unsigned long long)m & 0x8000000000000000ull)));
}

// Table of sin and cos at k 2^-8, k = 0 .. 805 (theta in [0, pi]), as Fx<62>.
constexpr int kFxTab = 806;
constexpr size_t kFxTabBytes = 2 * kFxTab * sizeof(fx64);

// sin and cos of th by angle addition from the nearest node: |d| <= 2^-9,
// sin d = d - d d2 (1/6 - d2/120) (d^7/5040 below 2^-75), cos d - 1 = -d2/2 + d2^2/24
// (d^6/720 below 2^-63).
__device__ __forceinline__ void fx_sincos(const fx64 *__restrict__ tab, Fx<61> th, Fx<62> &s, Fx<62> &c) {
    int k = (int)((th.m + (1ll << 52)) >> 53);
    k = k < 0 ? 0 : (k > kFxTab - 1 ? kFxTab - 1 : k);
    const Fx<70> d{fx_shl(th.m - fx_shl(k, 53), 9)};
    const Fx<62> sk{tab[2 * k]}, ck{tab[2 * k + 1]};
    const Fx<76> d2 = d * d;
    const int h2 = (int)(d2.m >> 28);                             // d2 in units of 2^-48
    const int h4 = (int)(((fx64)h2 * h2) >> 32);                  // d2^2 in units of 2^-64
    const fx64 q24 = ((fx64)h4 * 178956971) >> 32;                // d2^2/24, units of 2^-64
    const fx64 q120 = ((fx64)h4 * 35791394) >> 32;                // d2^2/120
    const Fx<76> cm{fx_shl(q24, 12) - (d2.m >> 1)};               // cos d - 1
    const Fx<65> sixth{6148914691236517205ll};                    // 1/6
    const Fx<77> t{(d2 * sixth).m - fx_shl(q120, 13)};            // d2/6 - d2^2/120
    const Fx<70> sd{d.m - ((d * t).m >> 13)};                     // sin d
    const Fx<68> ds = ck * sd + (sk * cm).dn<6>();
    const Fx<68> dc = (ck * cm).dn<6>() - sk * sd;
    s = Fx<62>{sk.m + ((ds.m + 32) >> 6)};
    c = Fx<62>{ck.m + ((dc.m + 32) >> 6)};
}

// 1/v for v in [0.2, 2.5] (Fx<60>): an FP32 seed y0 of 18 bits, e = 1 - v y0 exactly (its Q79
// product modulo 2^64), and y0 (1 + e + e^2 + e^3), which leaves e^4 < 2^-68.
template <int Q = 60>
__device__ __forceinline__ Fx<Q> fx_recip(Fx<60> v) {
    float f = (float)(int)(v.m >> 32), r;  // v 2^28
#ifdef __CUDA_ARCH__
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(f));
#else
    r = 1.0f / f;
#endif
    const int y0 = rint_small(r * 140737488355328.0f);  // 2^47 / (v 2^28) = 2^19 / v
    const unsigned long long lo = (unsigned long long)(unsigned)v.m * (unsigned)y0;
    const unsigned hi = (unsigned)((unsigned long long)v.m >> 32) * (unsigned)y0;
    const fx64 e = (fx64)(0ull - (lo + ((unsigned long long)hi << 32)));  // Q79
    const int eh = (int)(e >> 32);                   // Q47
    const fx64 e2 = (fx64)eh * eh;                   // Q94
    const fx64 e3 = (fx64)(int)(e2 >> 32) * eh;      // Q109
    const fx64 t = e + (e2 >> 15) + (e3 >> 30);      // Q79
    const fx64 y = (fx64)(int)(t >> 32) * y0 + (fx64)(((unsigned long long)(unsigned)t * (unsigned)y0) >> 32);  // Q66
    return Fx<Q>{fx_shl(y0, Q - 19) + (y >> (66 - Q))};
}

// The step's scale: exponents and spin.
struct FxScale {
    int e, kap, g, z;
    Fx<63> al;        // a 2^g / rho, |al| < 1/2
    Fx<64> nal2;      // minus its square, > -1/4
    unsigned klim, plim;  // bounds of the rates: hh |rate| < 1/4, below 2 (Q60) and 8 (P's, Q58), in units of 2^32
};
struct FxState {
    Fx<62> x;            // r / rho
    Fx<61> th;           // theta
    Fx<63> W, R, v, P;
};

// Negative (as an int) when m is outside [-lim 2^32, lim 2^32): the results of several checks are
// joined with |.
__device__ __forceinline__ unsigned fx_outside(fx64 m, unsigned lim) {
    const unsigned h = (unsigned)((unsigned long long)m >> 32);
    return (h + lim) | (lim - 1u - h);
}
// Negative when m < lo or m > hi (64-bit values no further apart than 2^62 from zero).
__device__ __forceinline__ unsigned fx_beyond(fx64 m, fx64 lo, fx64 hi) {
    const unsigned long long u = (unsigned long long)m;
    return (unsigned)((u - (unsigned long long)lo) >> 32) | (unsigned)(((unsigned long long)hi - u) >> 32);
}

// Minus the rates of (W, R, v, P) at a stage, from sin and cos of theta, in Q60 (P's in Q58). The
// metric is g = eta + q l l with eta the flat metric in oblate coordinates and l = (1, 1, 0,
// -a s^2), and the acceleration -g^{mu nu} F_nu with (D: the derivative along K, V = l K,
// T = K^r + q V)
//   F_t = V Dq - 2 q a s c K^th K^ph,
//   F_r = F_t - 2 a s c K^th K^ph - r (K^th^2 + s^2 K^ph^2) - V^2 dq/dr / 2,
//   F_ph = 2 r K^r s^2 K^ph + 2 (r^2 + a^2) s c K^th K^ph - 2 a s c K^th T - a s^2 F_t,
//   F_th = 2 r K^r K^th - a^2 s c K^th^2 - (r^2 + a^2) s c K^ph^2 + 2 a s c K^ph T - V^2 dq/dth / 2.
// In units of rho and 2^kap, with n for "minus":
//   isig = rho^2 / Sigma, qh = q rho / 2, Dr = (rho^2 / 2) dq/dr, del = (rho^2 / 2) Dq,
//   At = (rho^2 / 2) F_t, At2 = rho F_t, Fr = rho F_r, Fm = Fr - At2;
// and, in units of 2^-g for each factor of v, u, P or alpha,
//   Dt = (rho / 4) dq/dth 2^2g, Ap = F_ph 2^g = s J + 2 sa c v u 2^-g, F_th 2^g = F1 - sa c u P 2^(z - g).
// Every term in 1 / sin is written with P. A negative number in bad is a bound that failed.
__device__ __forceinline__ void fx_rates(const FxScale &S, const FxState &y, Fx<62> s, Fx<62> c, fx64 nk[4], unsigned &bad) {
    // counts of 64 and more (r above 2^22) leave a sign, as 63 does
    const int e1 = S.e - 1, g = S.g, g2 = 2 * g < 63 ? 2 * g : 63, g3 = 3 * g < 63 ? 3 * g : 63;
    // position terms
    const Fx<64> nal2 = S.nal2.over(g2);
    const Fx<60> na2s2 = nal2 * (s * s);                              // >= -1/4
    const Fx<60> sa = y.x * y.x - nal2.dn<4>();                       // <= 1.46
    const Fx<60> isig = fx_recip(sa + na2s2);                         // <= 4.94
    const Fx<61> qh = (y.x * isig).up<3>();                           // <= 2.23
    const Fx<61> q = qh.over(e1);
    const Fx<61> Dn{fx_shl((y.x * qh).m, 3) - (1ll << 61)};           // 2 x qh - 1: 0 .. 1
    const Fx<60> nDr = (isig * Dn).up<3>();                           // <= 4.94
    const Fx<64> nasc = (S.nal2 * (s * c)).up<4>();                   // 1/8
    const Fx<62> nDt = (nasc * (qh * isig).up<2>()).up<3>();          // 1.4
    const Fx<59> nA = na2s2.up<3>() * isig;                           // -a^2 s^2 / Sigma: > -1 where r > a (checked)
    const Fx<61> ai = (S.al * isig).up<2>();                          // 2.5
    const Fx<63> as = (S.al * s).up<2>();                             // 1/2
    // contractions with the momentum
    const Fx<63> u{fx_shl((s * y.P).m, S.z + 2)};
    const Fx<64> au = (S.al * u).up<2>();                             // 0.16
    const Fx<62> V = y.W.dn<1>() - s * au.over(g2);                   // 0.47
    const Fx<60> V2 = V * V;                                          // 0.22
    const Fx<64> V2e{fx_shl(V2.m, 3) >> e1};                          // V^2 / rho
    const Fx<63> cv = (c * y.v).up<2>(), cu = (c * u).up<2>();
    const Fx<62> E2{(cv * au).m >> g3};                               // 2 a s c K^th K^ph rho
    const Fx<62> v2 = y.v * y.v, uv2 = fx_dot(u, u, y.v, y.v);        // 0.2
    const Fx<61> ndel = fx_dot(y.R, nDr, y.v, nDt.dn<1>().twice().over(g3)).up<2>();  // 2.4
    const Fx<59> nAt = fx_dot(ndel, V, qh, E2);                       // 1.4
    const Fx<60> nAt2{fx_shl(nAt.m, 1) >> e1};
    const Fx<61> nFm = E2.dn<1>() + fx_dot(y.x, uv2.over(g2), -nDr, V2e).up<1>();  // 0.85
    const Fx<61> nFr = nAt2.up<1>() + nFm;                            // 2.2
    const Fx<62> T = y.R.dn<1>() + (q * V).up<3>();                   // 1.4
    const Fx<63> xR = (y.x * y.R).up<2>();                            // 0.35
    const Fx<61> G = fx_dot(xR, u, S.al, -((cv * T).up<2>().over(g))).twice();  // 0.65
    const Fx<62> scv = (sa * cv).up<3>().over(g);                     // 0.46
    const Fx<61> J = G + as * nAt2.up<2>();                           // 1.4
    const Fx<60> Ap = fx_dot(s, J.up<1>(), scv.twice(), u);           // 1.7
    // W and R: g^tt = -(1 + q), g^tr = q, g^rr = Delta / Sigma, g^rph = a / Sigma;
    // (r^2 + a^2) / Sigma = 1 + a^2 s^2 / Sigma
    const Fx<60> Y = fx_dot_fine(nA.up<3>(), nFr, ai, Ap.up<2>().over(g2)) - nFr.dn<1>();
    const Fx<60> nkW = nAt2 + Y, nkR = q * nFm.up<2>() + Y;
    // theta
    const Fx<64> acu = (S.al * cu).up<2>();                           // 0.16
    const Fx<61> F1 = fx_dot(xR.twice(), y.v, acu.twice().over(g), T) +
                      fx_dot(nasc.dn<1>(), v2.over(g3), nDt.twice().over(g), V2e);  // 0.9
    const fx64 cuP = (cu * y.P).m >> 2;                               // Q60
    const int zg = S.z - g, zl = zg > 0 ? zg : 0;
    const Fx<63> cz{fx_shl(cuP >> (zl - zg), zl + 3)};                // c u^2 / s, < 1
    const Fx<60> npi{fx_shl(nA.m, 1) - (1ll << 60)};                  // -(r^2 + a^2) / Sigma
    const Fx<60> nkv = fx_dot_fine(isig, F1.up<2>(), npi, cz);
    // phi: (isig / s) (2 sa c v P 2^-g + (al s Fm + G) / 2^z)
    const fx64 sm = (unsigned long long)s.m < 1ull << 62 ? s.m : (1ll << 62) - 1;  // (a negative one fails below)
    const int zs = fx_clz((unsigned long long)(sm | 1)) - 2;          // s 2^zs in [1/2, 1)
    const Fx<61> isn = fx_recip<61>(Fx<60>{fx_shl(sm, zs) >> 2});
    const Fx<60> B = (scv * y.P).twice() + (G - fx_fine<1>(as, nFm)).dn<1>().over(S.z);
    const Fx<58> nkP = fx_fine<2>(isig, B.up<3>()) * isn;
    nk[0] = nkW.m;
    nk[1] = nkR.m;
    nk[2] = nkv.m;
    nk[3] = fx_shl(nkP.m, zs);
    // bounds: the momentum (5/16), the position, sin >= 2^-10, c u^2 / s < 1, B < 3/4, and the rates
    bad |= fx_outside(y.W.m, 0x28000000u) | fx_outside(y.R.m, 0x28000000u) | fx_outside(y.v.m, 0x28000000u) |
           fx_outside(y.P.m, 0x28000000u) | fx_outside(u.m, 0x28000000u);
    bad |= fx_beyond(y.x.m, 2075258708292324556ll, 5072854620270126694ll);  // 0.45, 1.1
    bad |= fx_beyond(s.m, 1ll << 52, (1ll << 62) + (1ll << 40));
    bad |= fx_outside(cuP, 1u << (28 - zl)) | fx_outside(B.m, 3u << 26) | fx_outside(nA.m, 1u << 27);
    bad |= fx_outside(nkW.m, S.klim) | fx_outside(nkR.m, S.klim) | fx_outside(nkv.m, S.klim) | fx_outside(nkP.m, S.plim >> zs);
}

// One classic RK4 step of size h from y = (r, theta, phi, W, K^r, K^theta, K^phi) to out. Returns
// false (out undefined) where the step is outside the form's bounds.
__device__ __forceinline__ bool fx_step(const fx64 *__restrict__ tab, double a, double h, const double y[7], double out[7]) {
    auto ex = [](double d) { return (int)(((unsigned long long)__double_as_longlong(d) >> 52) & 0x7ffull) - 1022; };
    FxScale S;
    S.e = ex(y[0]);
    const int hx0 = ex(h);
    unsigned bad = (unsigned)(S.e - 1) | (unsigned)(40 - S.e) | (unsigned)(2 - ex(y[1]));
    S.e = S.e < 1 ? 1 : (S.e > 40 ? 40 : S.e);
    FxState b, t;
    b.x.m = fx_from(y[0], 62 - S.e);
    b.th.m = fx_from(y[1], 61);
    t = b;
    int hx = 0;
    Fx<62> hm{0};  // hh = hm 2^hx with hm in [1/2, 1)
    // hh k (or hh k / 2) as a sum's term: the product, then a shift
    auto scaled = [](fx64 p, int n) { return fx_shl(p >> (n < 0 ? -n : 0), n < 0 ? 0 : n); };
    fx64 nk[4], SK[4], SP[3];
#pragma unroll 1
    for (int st = 0; st < 4; st++) {
        bad |= fx_beyond(t.th.m, 0, 805ll << 53);
        Fx<62> s, c;
        fx_sincos(tab, t.th, s, c);
        if (st == 0) {
            // the largest of |W|, |R|, rho |K^theta|, rho sin |K^phi| below 2^(kap - 2), and the
            // last two below 2^(kap - g - 2)
            const int ep = ex(y[6]) + S.e;
            const int x1 = ex(y[4]), x2 = ex(y[5]) + S.e, x3 = ep + 2 - fx_clz((unsigned long long)(s.m | 1));
            const int xt = x2 > x3 ? x2 : x3;
            int kap = ex(y[3]);
            kap = kap > x1 ? kap : x1;
            kap = (kap > xt ? kap : xt) + 2;
            S.g = kap - 2 - xt;
            S.g = S.g < S.e - 1 ? S.g : S.e - 1;
            const int kt = kap - S.g;
            S.z = ep + 2 - kt;
            S.z = S.z < 0 ? 0 : S.z;
            hx = hx0 + kap - S.e;
            bad |= (unsigned)(200 - kap) | (unsigned)(kap + 200) | (unsigned)(11 - S.z) | (unsigned)(3 - hx) |
                   (unsigned)(hx + 20) | fx_beyond(s.m, 1ll << 52, (1ll << 62) + (1ll << 40));
            if ((int)bad < 0) return false;
            S.kap = kap;
            S.klim = 1u << (26 - (hx < -3 ? -3 : hx));
            S.plim = 1u << (24 - (hx < -5 ? -5 : hx));
            b.W.m = fx_from(y[3], 63 - kap);
            b.R.m = fx_from(y[4], 63 - kap);
            b.v.m = fx_from(y[5], 63 - kt + S.e);
            b.P.m = fx_from(y[6], 63 - kt - S.z + S.e);
            S.al.m = fx_from(a, 63 - S.e + S.g);
            S.nal2 = -((S.al * S.al).up<2>());
            t = b;
            hm.m = fx_from(h, 62 - hx0);
        }
        fx_rates(S, t, s, c, nk, bad);
        // sums of the rates, halved: k1 + 2 k2 + 2 k3 + k4 and k1 + k2 + k3
        if (st == 0) {
#pragma unroll
            for (int i = 0; i < 4; i++) SK[i] = nk[i] >> 1;
#pragma unroll
            for (int i = 0; i < 3; i++) SP[i] = nk[i + 1] >> 1;
        } else if (st == 3) {
#pragma unroll
            for (int i = 0; i < 4; i++) SK[i] += nk[i] >> 1;
            break;
        } else {
#pragma unroll
            for (int i = 0; i < 4; i++) SK[i] += nk[i];
#pragma unroll
            for (int i = 0; i < 3; i++) SP[i] += nk[i + 1] >> 1;
        }
        // the next stage: positions advance with this stage's momentum
        const int hs = st < 2 ? hx - 1 : hx;
        t.x.m = b.x.m + scaled(fx_mulhi(hm.m, t.R.m), hs + 1);
        t.th.m = b.th.m + scaled(fx_mulhi(hm.m, t.v.m), hs - S.g);
        t.W.m = b.W.m - scaled(fx_mulhi(hm.m, nk[0]), hs + 5);
        t.R.m = b.R.m - scaled(fx_mulhi(hm.m, nk[1]), hs + 5);
        t.v.m = b.v.m - scaled(fx_mulhi(hm.m, nk[2]), hs + 5);
        t.P.m = b.P.m - scaled(fx_mulhi(hm.m, nk[3]), hs + 7);
    }
    if ((int)bad < 0) return false;
    // position' = position + h K + (h^2 / 6) (k1 + k2 + k3), K' = K + (h / 6) (k1 + 2 k2 + 2 k3 + k4);
    // the halved sums in Q60 are the sums in Q59 (P's in Q57), and the products two bits finer
    const Fx<65> sixth{6148914691236517205ll};
    const Fx<64> h6 = (hm * sixth).up<1>();
    out[0] = y[0] + fx_to(fx_mulhi(hm.m, b.R.m - scaled(fx_mulhi(h6.m, SP[0]), hx + 4)), 61 - hx - S.e);
    out[1] = y[1] + fx_to(fx_mulhi(hm.m, b.v.m - scaled(fx_mulhi(h6.m, SP[1]), hx + 4)), 61 - hx + S.g);
    out[2] = y[2] + fx_to(fx_mulhi(hm.m, b.P.m - scaled(fx_mulhi(h6.m, SP[2]), hx + 6)), 61 - hx - S.z + S.g);
    out[3] = y[3] - fx_to(fx_mulfine<2>(h6.m, SK[0]), 61 - hx - S.kap);
    out[4] = y[4] - fx_to(fx_mulfine<2>(h6.m, SK[1]), 61 - hx - S.kap);
    out[5] = y[5] - fx_to(fx_mulfine<2>(h6.m, SK[2]), 61 - hx - S.kap + S.g + S.e);
    out[6] = y[6] - fx_to(fx_mulfine<2>(h6.m, SK[3]), 59 - hx - S.kap - S.z + S.g + S.e);
    return true;
}

}  // namespace prt
