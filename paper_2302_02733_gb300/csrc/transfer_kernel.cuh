// The transfer along the saved geodesics, from the far end back to the camera. At every saved
// state the screen legs are parallel-transported (Heun, connection from the saved K) and the
// plasma is evaluated, and if the point emits, the Stokes vector is projected onto the fluid screen
// and takes the exact constant-coefficient step. Instantiated for the FP64 and the mixed (FP32
// transfer) forms.
//
// Only the Stokes vector is a chain along the ray: the plasma, tetrad, coefficients and the change
// of screen from one emitting point to the next depend on the geometry alone. So the transfer is
// two kernels: points_kernel, one warp per ray and one lane per saved state, 32 at a time, replaces
// each state by its step's record (XRec); chain_kernel, one lane per ray, applies the records in
// turn. transfer_kernel, one lane per ray for both, runs where the FP64 records have no room. Transfers
// with it and with the two kernels: FP64 ADAF 64^2 39.5 and 9.5 ms, torus 126 x 130 59 and 23, 200^2 85 and
// 50, 300^2 132 and 104, kappa 20^2 223 and 11; mixed torus 64^2 5.8 and 1.5, 300^2 12 and 6.0, 1024^2 69 and
// 61.
#pragma once
#include <cuda.h>

#include "surrogate.cuh"
#include "tc.cuh"
#include "transfer.cuh"

namespace prt {

// The FP32 form reads the FP64 path with d2f_int (ffloat.cuh): integer operations only.
template <typename R>
__device__ __forceinline__ R to_real(double d);
template <>
__device__ __forceinline__ double to_real<double>(double d) {
    return d;
}
template <>
__device__ __forceinline__ float to_real<float>(double d) {
    return d2f_int(d);
}

// o = T v for a 4x4 matrix
template <typename R>
__device__ __forceinline__ void matvec4(const R T[4][4], const R v[4], R o[4]) {
#pragma unroll
    for (int m = 0; m < 4; m++) o[m] = T[m][0] * v[0] + T[m][1] * v[1] + T[m][2] * v[2] + T[m][3] * v[3];
}

// Heun step of a screen leg held as base + increment, E = eo + u: with a = T(x_{n+1}) E known
// from the previous point and T0 = T(x_n), v = E + h a and E gains (h/2)(a + T0 v). Only the
// increment u changes, so E - e (needed by the compensated re-projection) stays exact.
template <typename R>
__device__ __forceinline__ void heun_leg(const R eo[4], R u[4], const R a[4], const R T0[4][4], R h) {
    R v[4];
#pragma unroll
    for (int m = 0; m < 4; m++) v[m] = (eo[m] + u[m]) + h * a[m];
    R hh = R(0.5) * h;
#pragma unroll
    for (int m = 0; m < 4; m++)
        u[m] += hh * (a[m] + T0[m][0] * v[0] + T0[m][1] * v[1] + T0[m][2] * v[2] + T0[m][3] * v[3]);
}

// An opaque copy: the value is rounded here, in every kernel, and no sum made of it later contracts
// the product it came from. The values that pass from the geometry of a point to the Stokes chain
// go through it, so that both transfers give the same bits.
__device__ __forceinline__ float pinned(float x) {
    asm volatile("" : "+f"(x));
    return x;
}
__device__ __forceinline__ double pinned(double x) {
    asm volatile("" : "+d"(x));
    return x;
}

// What one saved state does to the Stokes vector: the change of screen D on arrival (n' - n =
// D n + n D^T + D n D^T), then the constant-coefficient step's optical depths and emission (J
// with j_U = 0). tau = -infinity marks a state that does not emit.
template <typename R>
struct XRec {
    R d11, d12, d21, d22, tau, aQ, aV, rQ, rV, J0, J1, J3;
};

// FP64: the second parts of the states' records (4 doubles each) lie behind the arena blocks that the
// chunk's rays took, in what they left of their budget; NULL where that is less than half of what they took
// (the one-lane kernel then runs). 12 of 20 blocks are usual at the default step.
__device__ __forceinline__ double *record_tail(const XferArgs &p) {
    const unsigned long long used = p.ctr->arena_next;
    return 3 * used <= 2 * (unsigned long long)p.arena.nblocks ? reinterpret_cast<double *>(p.arena.states + used * kBlockStates) : nullptr;
}

// The 2x2 matrix C_{ij} = f_i . E_j from the screen (E1, E2) to the screen (f1, f2) given as lowered
// legs, used once, at the camera: C = (c11, c12, c21, c22).
template <typename R>
__device__ __forceinline__ void screen_matrix(const R f1[4], const R f2[4], const R E1[4], const R E2[4], R C[4]) {
    C[0] = pinned(f1[0] * E1[0] + f1[1] * E1[1] + f1[2] * E1[2] + f1[3] * E1[3]);
    C[1] = pinned(f1[0] * E2[0] + f1[1] * E2[1] + f1[2] * E2[2] + f1[3] * E2[3]);
    C[2] = pinned(f2[0] * E1[0] + f2[1] * E1[1] + f2[2] * E1[2] + f2[3] * E1[3]);
    C[3] = pinned(f2[0] * E2[0] + f2[1] * E2[1] + f2[2] * E2[2] + f2[3] * E2[3]);
}

// Stokes (I, Q, U, V) re-expressed on another screen: n' = C n C^T.
template <typename R>
__device__ __forceinline__ void reproject(const R C[4], R S[4]) {
    const R c11 = C[0], c12 = C[1], c21 = C[2], c22 = C[3];
    R n11 = R(0.5) * (S[0] + S[1]), n22 = R(0.5) * (S[0] - S[1]), nr = R(0.5) * S[2];
    R m11 = c11 * c11 * n11 + R(2) * c11 * c12 * nr + c12 * c12 * n22;
    R m22 = c21 * c21 * n11 + R(2) * c21 * c22 * nr + c22 * c22 * n22;
    R mr = c11 * c21 * n11 + (c11 * c22 + c12 * c21) * nr + c12 * c22 * n22;
    R det = c11 * c22 - c12 * c21;
    S[0] = m11 + m22;
    S[1] = m11 - m22;
    S[2] = R(2) * mr;
    S[3] = det * S[3];
}

// The change of screen D from the transported legs E_k = eo_k + u_k to the new fluid screen
// (e1, e2), lowered l1, l2. The new coefficients are
// n' = C n C^T with C = G^{-1} A, A_ik = l_i . E_k and G_ij = l_i . e_j: the dual basis of
// (e1, e2), so the rounding of their norms does not scale the intensity. Writing
// E_k = e_k + Delta_k with Delta_k = (eo_k - e_k) + u_k (exact differences of nearby legs plus
// the transport increment) gives C = 1 + D, D = G^{-1} Lambda, Lambda_ik = l_i . Delta_k.
template <typename R>
__device__ __forceinline__ void screen_change(const R l1[4], const R l2[4], const R e1[4], const R e2[4],
                                              const R eo1[4], const R eo2[4], const R u1[4], const R u2[4], XRec<R> &x) {
    R L11 = 0, L12 = 0, L21 = 0, L22 = 0, g11 = 0, g12 = 0, g21 = 0, g22 = 0;
#pragma unroll
    for (int i = 0; i < 4; i++) {
        R d1 = (eo1[i] - e1[i]) + u1[i];
        R d2 = (eo2[i] - e2[i]) + u2[i];
        L11 += l1[i] * d1;
        L12 += l1[i] * d2;
        L21 += l2[i] * d1;
        L22 += l2[i] * d2;
        g11 += l1[i] * e1[i];
        g12 += l1[i] * e2[i];
        g21 += l2[i] * e1[i];
        g22 += l2[i] * e2[i];
    }
    R idet = R(1) / (g11 * g22 - g12 * g21);
    x.d11 = pinned((g22 * L11 - g12 * L21) * idet), x.d12 = pinned((g22 * L12 - g12 * L22) * idet);
    x.d21 = pinned((g11 * L21 - g21 * L11) * idet), x.d22 = pinned((g11 * L22 - g21 * L12) * idet);
}

// Stokes on the new screen as a compensated increment: n' - n = D n + n D^T + D n D^T; V scales by
// det C = 1 + tr D + det D. The change is small where the screen turns slowly and is added to
// (S, Slo) without rounding loss.
template <typename R>
__device__ __forceinline__ void reproject_comp(const XRec<R> &x, R S[4], R Slo[4]) {
    const R d11 = x.d11, d12 = x.d12, d21 = x.d21, d22 = x.d22;
    R n11 = R(0.5) * (S[0] + S[1]), n22 = R(0.5) * (S[0] - S[1]), nr = R(0.5) * S[2];
    R x11 = d11 * n11 + d12 * nr, x12 = d11 * nr + d12 * n22;
    R x21 = d21 * n11 + d22 * nr, x22 = d21 * nr + d22 * n22;
    R dn11 = R(2) * x11 + (x11 * d11 + x12 * d12);
    R dn22 = R(2) * x22 + (x21 * d21 + x22 * d22);
    R dnr = (x12 + x21) + (x11 * d21 + x12 * d22);
    R dV = pinned(((d11 + d22) + (d11 * d22 - d12 * d21)) * S[3]);
    two_sum_add(S[0], Slo[0], dn11 + dn22);
    two_sum_add(S[1], Slo[1], dn11 - dn22);
    two_sum_add(S[2], Slo[2], R(2) * dnr);
    two_sum_add(S[3], Slo[3], dV);
}

// The screen legs leaving a state: eo + u (base, transport increment), a1, a2: T E of the legs there;
// basis: whether a state at or before it (from the far end) emits.
template <typename R>
struct XLegs {
    R eo1[4], eo2[4], u1[4], u2[4], a1[4], a2[4];
    bool basis;
};

// The Stokes chain of one ray. S + Slo: Stokes / nu^3 (invariant) as a value and its compensation;
// tau, phi: optical and Faraday depths with their Kahan compensations.
template <typename R>
struct XChain {
    R S[4], Slo[4];
    R tau, tauc, phi, phic;
    __device__ __forceinline__ void reset() {
#pragma unroll
        for (int i = 0; i < 4; i++) S[i] = Slo[i] = R(0);
        tau = tauc = phi = phic = R(0);
    }
    // Every input is pinned here, in one order: the compiler orders commutative operands by where
    // they come from, and with them which of two products a sum contracts.
    __device__ __forceinline__ void apply(const XRec<R> &r) {
        const XRec<R> x = {pinned(r.d11), pinned(r.d12), pinned(r.d21), pinned(r.d22), pinned(r.tau), pinned(r.aQ),
                           pinned(r.aV),  pinned(r.rQ),  pinned(r.rV),  pinned(r.J0),  pinned(r.J1),  pinned(r.J3)};
#pragma unroll
        for (int i = 0; i < 4; i++) S[i] = pinned(S[i]), Slo[i] = pinned(Slo[i]);
        reproject_comp(x, S, Slo);
#pragma unroll
        for (int i = 0; i < 4; i++) S[i] = pinned(S[i]), Slo[i] = pinned(Slo[i]);
        const R J[4] = {x.J0, x.J1, R(0), x.J3};
        substep(x.tau, x.aQ, x.aV, x.rQ, x.rV, J, S, Slo);
#pragma unroll
        for (int i = 0; i < 4; i++) S[i] = pinned(S[i]), Slo[i] = pinned(Slo[i]);
        kahan_add(tau, tauc, x.tau);
        kahan_add(phi, phic, x.rV);
    }
};

// Per-lane transfer state of one ray, where one lane does both.
template <typename R>
struct XLane : XLegs<R>, XChain<R> {
    __device__ __forceinline__ void reset() {
        XChain<R>::reset();
        this->basis = false;
    }
};

// The surrogate's maps (surrogate.cuh) in the transfer's precision R, from the tetrad's sin and
// cos of the field angle (sth >= 0) instead of the angle, for the FP32 render: the prefactors are
// written as in the thermal fits (nu_B / nu and e^2 / (m c) grouped) so every intermediate
// stays within FP32 range.
template <typename R>
struct SurPrefR {
    R Pj, PjV, Pa, PaV, PrQ, PrV, sgn;
};

template <typename R>
__device__ __forceinline__ SurPrefR<R> sur_prefactors_r(R ne, R Te, R B, R nu, R sth, R cth) {
    typedef Mth<R> F;
    const R cB = R(kQe / (2.0 * kPi * kMe * kC));             // nu_B / B
    const R cQ2 = R(kQe * kQe / (kMe * kC));                  // e^2 / (m c)
    const R cJ = R(kQe * kQe / (2.0 * 1.7320508075688772 * kC));
    SurPrefR<R> p;
    R as = fabs(sth), ac = fabs(cth);
    R rb = cB * B / nu;
    R cot = as > R(0) ? ac / as : R(0);
    p.Pj = cJ * ne * nu / (Te * Te);
    p.PjV = p.Pj * (R(4) / (R(3) * Te)) * cot;
    p.Pa = cQ2 * ne / (R(4.0 * 1.7320508075688772) * nu * Te * Te * Te);
    p.PaV = p.Pa * cot;
    R X = Te * F::sqrt_(R(1.4142135623730951) * as * R(1e3) * rb);
    R f = shcherbakov_fX(X);
    p.PrQ = cQ2 * ne * rb * rb / nu * sth * sth * f;
    p.PrV = R(2) * cQ2 * ne * rb / nu * ac * (R(1) - R(0.11) * F::log1p_(R(0.035) * X));
    p.sgn = cth < R(0) ? R(-1) : R(1);
    return p;
}

template <typename R>
__device__ __forceinline__ void sur_features_r(R Te, R B, R nu, R sth, R cth, R kappa, float f[4]) {
    typedef Mth<R> F;
    const R cB = R(kQe / (2.0 * kPi * kMe * kC));
    R tf = F::atan2_(sth, fabs(cth));  // theta_B folded into [0, pi/2]
    f[0] = (float)(-F::log_(R(1.5) * cB * B / nu * sth * Te * Te));
    f[1] = (float)tf;
    f[2] = (float)F::log_(Te);
    f[3] = (float)kappa;
}

template <typename R>
__device__ __forceinline__ void sur_expand_r(const SurPrefR<R> &p, const float y[8], R c[8]) {
    typedef Mth<R> F;
    c[0] = p.Pj * F::exp_(R(y[0]));
    c[1] = p.Pj * F::exp_(R(y[1]));
    c[2] = p.sgn * p.PjV * F::exp_(R(y[2]));
    c[3] = p.Pa * F::exp_(R(y[3]));
    c[4] = p.Pa * F::exp_(R(y[4]));
    c[5] = p.sgn * p.PaV * F::exp_(R(y[5]));
    c[6] = p.PrQ * F::exp_(R(y[6]));
    c[7] = p.sgn * p.PrV * F::exp_(R(y[7]));
    R pj = F::sqrt_(c[1] * c[1] + c[2] * c[2]);
    if (pj > c[0] && pj > R(0)) {
        c[1] *= c[0] / pj;
        c[2] *= c[0] / pj;
    }
    R pa = F::sqrt_(c[4] * c[4] + c[5] * c[5]);
    if (pa > c[3] && pa > R(0)) {
        c[4] *= c[3] / pa;
        c[5] *= c[3] / pa;
    }
}

// Coefficients of an emitting point for kappa electrons: CM 1 by quadrature, CM 2 from the
// surrogate's outputs for this saved state (quadrature outside the network's box).
template <typename R, int CM>
__device__ __forceinline__ void kappa_point_coeffs(const XferArgs *pa, long long st, const Model &mdl,
                                                   const Plasma<R> &pl, R w, R sth, R cth, R nu_obs, R cf[8]) {
    typedef Mth<R> F;
    if (CM == 2) {  // the network, in R, inside its box
        float f[4], xn[4];
        sur_features_r<R>(pl.Te, pl.B, w * nu_obs, sth, cth, R(mdl.kappa), f);
        bool in = true;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            float u = (f[j] - pa->sur_lo[j]) / (pa->sur_hi[j] - pa->sur_lo[j]);
            in &= u >= 0.0f && u <= 1.0f;
            xn[j] = 2.0f * u - 1.0f;
        }
        if (in) {
            float phi[kSurBasis], y[8];
            sur_basis(xn, phi);
            const long long row = pa->sur_row ? (long long)pa->sur_row[st] : st;
            const float *nm = pa->sur_norm, *yh = pa->sur_y + 8 * row;
#pragma unroll
            for (int k = 0; k < 8; k++) {
                float b = 0.f;
                for (int q = 0; q < kSurBasis; q++) b += nm[16 + k * kSurBasis + q] * phi[q];
                y[k] = b + nm[k] + nm[8 + k] * yh[k];
            }
            sur_expand_r<R>(sur_prefactors_r<R>(pl.ne, pl.Te, pl.B, w * nu_obs, sth, cth), y, cf);
            if (!(cf[0] > F::jflush))
#pragma unroll
                for (int k = 0; k < 6; k++) cf[k] = R(0);
            return;
        }
    }
    // quadrature (CM 1, or CM 2 outside the network's box), in FP64: the exact grade for the
    // FP64 form, the tabulated one for the FP32 forms
    double thB = atan2((double)sth, (double)cth), nu = (double)(w * nu_obs);
    double cd[8];
    kappa_coeffs_quad<sizeof(R) == 8>(pa->kt, (double)pl.ne, (double)pl.Te, (double)pl.B, nu, thB, mdl.kappa, cd);
#pragma unroll
    for (int k = 0; k < 8; k++) cf[k] = R(cd[k]);
    if (!(cf[0] > F::jflush))  // as for the thermal fits: no relative precision left
#pragma unroll
        for (int k = 0; k < 6; k++) cf[k] = R(0);
}

// pre (optional): the grid cell of this state and its interpolated primitives, fetched by the
// caller (the staged transfer); a null cell pointer means the state lies outside the grid.
template <typename R>
struct PreFetch {
    const GridCell<R> *cell;
    const R *P;
};

// What a saved state (q0, q1) contributes by itself: its metric, step, connection and, where the
// point emits (valid), the fluid screen and the radiative step of its record.
template <typename R>
struct XPoint {
    KS<R> m;
    R K[4], h;
    bool flip;  // the step to this state's far neighbour crossed the polar axis
    bool valid;
    R e1[4], e2[4];
};

template <typename R, int CM = 0, bool PRE = false>
__device__ __forceinline__ void xfer_eval(const Camera &c, const Model &mdl, const double4_32a &q0,
                                          const double4_32a &q1, const R *sgw, XPoint<R> &P, XRec<R> &x,
                                          const XferArgs *pa = nullptr, long long st = 0,
                                          PreFetch<R> pre = PreFetch<R>{nullptr, nullptr}) {
    const R a = pick<R>(c.a, c.f_a);
    R r = to_real<R>(q0.x), th = to_real<R>(q0.y);
    P.K[0] = to_real<R>(q0.w), P.K[1] = to_real<R>(q1.x), P.K[2] = to_real<R>(q1.y), P.K[3] = to_real<R>(q1.z);
    R hs = to_real<R>(q1.w);
    P.h = fabs(hs);
    P.flip = hs < R(0);
    KS<R> &m = P.m;
    m.eval(a, r, th);
    Plasma<R> pl;
    if (PRE) {
        pl.valid = false;
        if (pre.cell) grid_state(mdl.grid, m, *pre.cell, pre.P, pl);
    } else if (mdl.kind == 1) {
        adaf_plasma(mdl.adaf, a, m, r, pl);
    } else {
        grid_plasma(mdl.grid, m, q0.x, q0.y, q0.z, pl);
    }
    P.valid = pl.valid;
    if (!pl.valid) return;
    R w, sth, cth;
    fluid_tetrad(m, P.K, pl.u, pl.b, P.e1, P.e2, w, sth, cth);
    w = pinned(w), sth = pinned(sth), cth = pinned(cth);
#pragma unroll
    for (int i = 0; i < 4; i++) P.e1[i] = pinned(P.e1[i]), P.e2[i] = pinned(P.e2[i]);
    R cf[8];
    if (CM == 0)
        thermal_coeffs(pl.ne, pl.Te, pl.B, w * pick<R>(c.nu_obs, c.f_nu_obs), sth, cth, sgw, cf);
    else
        kappa_point_coeffs<R, CM>(pa, st, mdl, pl, w, sth, cth, pick<R>(c.nu_obs, c.f_nu_obs), cf);
    // invariant form: S holds I/nu^3, so the step takes J/w^3 and the same M
    R ds = w * P.h * pick<R>(c.L_unit, c.f_L_unit);
    R jds = R(1) / (w * w * w) * ds;
    x.tau = pinned(cf[3] * ds), x.aQ = pinned(cf[4] * ds), x.aV = pinned(cf[5] * ds);
    x.rQ = pinned(cf[6] * ds), x.rV = pinned(cf[7] * ds);
    x.J0 = pinned(cf[0] * jds), x.J1 = pinned(cf[1] * jds), x.J3 = pinned(cf[2] * jds);
}

// The legs leaving a state from those leaving its far neighbour (L, updated): transported, and where
// the state emits replaced by its fluid screen, the change into x. T0: the connection there.
template <typename R>
__device__ __forceinline__ void xfer_link(const XPoint<R> &P, const R T0[4][4], XLegs<R> &L, XRec<R> &x) {
    if (L.basis) {
        if (P.flip) {  // that step crossed the polar axis: bring n+1 into this chart
            L.eo1[2] = -L.eo1[2];
            L.eo2[2] = -L.eo2[2];
            L.u1[2] = -L.u1[2];
            L.u2[2] = -L.u2[2];
            L.a1[2] = -L.a1[2];
            L.a2[2] = -L.a2[2];
        }
        heun_leg(L.eo1, L.u1, L.a1, T0, P.h);
        heun_leg(L.eo2, L.u2, L.a2, T0, P.h);
#pragma unroll
        for (int i = 0; i < 4; i++) L.u1[i] = pinned(L.u1[i]), L.u2[i] = pinned(L.u2[i]);
    }
    if (P.valid) {
        x.d11 = x.d12 = x.d21 = x.d22 = R(0);
        if (L.basis) {
            R l1[4], l2[4];
            P.m.lower(P.e1, l1);
            P.m.lower(P.e2, l2);
#pragma unroll
            for (int i = 0; i < 4; i++) l1[i] = pinned(l1[i]), l2[i] = pinned(l2[i]);
            screen_change(l1, l2, P.e1, P.e2, L.eo1, L.eo2, L.u1, L.u2, x);
        }
    }
}

// The legs leaving an emitting state: its fluid screen. pinned: another lane takes them up.
template <typename R>
__device__ __forceinline__ void xfer_screen(const XPoint<R> &P, const R T0[4][4], XLegs<R> &L) {
#pragma unroll
    for (int i = 0; i < 4; i++) {
        L.eo1[i] = P.e1[i];
        L.eo2[i] = P.e2[i];
        L.u1[i] = L.u2[i] = R(0);
    }
    matvec4(T0, P.e1, L.a1);
    matvec4(T0, P.e2, L.a2);
#pragma unroll
    for (int i = 0; i < 4; i++) L.a1[i] = pinned(L.a1[i]), L.a2[i] = pinned(L.a2[i]);
    L.basis = true;
}
// and those leaving a state that does not: T E of the transported ones
template <typename R>
__device__ __forceinline__ void xfer_pass(const R T0[4][4], XLegs<R> &L) {
    R E1[4], E2[4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
        E1[i] = L.eo1[i] + L.u1[i];
        E2[i] = L.eo2[i] + L.u2[i];
    }
    matvec4(T0, E1, L.a1);
    matvec4(T0, E2, L.a2);
#pragma unroll
    for (int i = 0; i < 4; i++) L.a1[i] = pinned(L.a1[i]), L.a2[i] = pinned(L.a2[i]);
}

// One saved state of the walk toward the camera on a lane of its own. m returns the metric at the
// state. Returns whether the point emits.
template <typename R, int CM = 0, bool PRE = false>
__device__ __forceinline__ bool xfer_point(const Camera &c, const Model &mdl, const double4_32a &q0,
                                           const double4_32a &q1, const R *sgw, XLane<R> &Ln, KS<R> &m,
                                           const XferArgs *pa = nullptr, long long st = 0,
                                           PreFetch<R> pre = PreFetch<R>{nullptr, nullptr}) {
    XPoint<R> P;
    XRec<R> x;
    xfer_eval<R, CM, PRE>(c, mdl, q0, q1, sgw, P, x, pa, st, pre);
    m = P.m;
    if (!Ln.basis && !P.valid) return false;
    R T0[4][4];
    connection_T(P.m, P.K, T0);
    xfer_link(P, T0, Ln, x);
    if (P.valid) {
        xfer_screen(P, T0, Ln);
        Ln.apply(x);
    } else {
        xfer_pass(T0, Ln);
    }
    return P.valid;
}

// At the camera (the last state, metric m): the matrix from the legs to the image basis of pixel
// (ix, iy); zero for a ray that nothing emitted on.
template <typename R>
__device__ __forceinline__ void camera_matrix(const Camera &c, const KS<R> &m, int ix, int iy, const XLegs<R> &Ln, R C[4]) {
    C[0] = C[1] = C[2] = C[3] = R(0);
    if (Ln.basis) {
        // camera screen: x along e_phi, y along -e_theta, each normal to the ray
        R X[4], Y[4];
        if constexpr (sizeof(R) == 4) {
            // the FP32 form: the camera frame from the host (c.f_e), the sky direction in float,
            // with no FP64 instruction (this runs once per ray, on a lane of its own)
            float px = (i2f_small(ix) + 0.5f) * c.f_pix - 0.5f * (c.f_pix * i2f_small(c.nx));
            float py = (i2f_small(iy) + 0.5f) * c.f_pix - 0.5f * (c.f_pix * i2f_small(c.ny));
            float al = px / c.f_r_cam, be = py / c.f_r_cam;
            float n = rsqrtf(1.0f + al * al + be * be);
            float s[3] = {-n, -be * n, al * n};
            float xh[3] = {-s[2] * s[0], -s[2] * s[1], 1.0f - s[2] * s[2]};
            float nx = rsqrtf(xh[0] * xh[0] + xh[1] * xh[1] + xh[2] * xh[2]);
            float yh[3] = {s[1] * s[0], -1.0f + s[1] * s[1], s[1] * s[2]};
#pragma unroll
            for (int k = 0; k < 3; k++) xh[k] *= nx;
            float yx = yh[0] * xh[0] + yh[1] * xh[1] + yh[2] * xh[2];
#pragma unroll
            for (int k = 0; k < 3; k++) yh[k] -= yx * xh[k];
            float ny = rsqrtf(yh[0] * yh[0] + yh[1] * yh[1] + yh[2] * yh[2]);
#pragma unroll
            for (int mu = 0; mu < 4; mu++) {
                X[mu] = xh[0] * c.f_e[0][mu] + xh[1] * c.f_e[1][mu] + xh[2] * c.f_e[2][mu];
                Y[mu] = ny * (yh[0] * c.f_e[0][mu] + yh[1] * c.f_e[1][mu] + yh[2] * c.f_e[2][mu]);
            }
        } else {
            const double(&e)[4][4] = c.e;
            double s[3];
            sky_direction(c, ix, iy, s);
            double xh[3] = {-s[2] * s[0], -s[2] * s[1], 1.0 - s[2] * s[2]};
            double nx = rsqrt(xh[0] * xh[0] + xh[1] * xh[1] + xh[2] * xh[2]);
            double yh[3] = {s[1] * s[0], -1.0 + s[1] * s[1], s[1] * s[2]};
            double yx = yh[0] * xh[0] * nx + yh[1] * xh[1] * nx + yh[2] * xh[2] * nx;
            for (int k = 0; k < 3; k++) {
                xh[k] *= nx;
                yh[k] -= yx * xh[k];
            }
            double ny = rsqrt(yh[0] * yh[0] + yh[1] * yh[1] + yh[2] * yh[2]);
#pragma unroll
            for (int mu = 0; mu < 4; mu++) {
                X[mu] = R(xh[0] * e[1][mu] + xh[1] * e[2][mu] + xh[2] * e[3][mu]);
                Y[mu] = R(ny * (yh[0] * e[1][mu] + yh[1] * e[2][mu] + yh[2] * e[3][mu]));
            }
        }
        R lx[4], ly[4], E1[4], E2[4];
        m.lower(X, lx);
        m.lower(Y, ly);
#pragma unroll
        for (int i = 0; i < 4; i++) {
            E1[i] = Ln.eo1[i] + Ln.u1[i];
            E2[i] = Ln.eo2[i] + Ln.u2[i];
        }
        screen_matrix(lx, ly, E1, E2, C);
    }
}

// Project the chain's Stokes vector onto the image basis and write pixel (ix, iy) of out (and of
// depth, if given).
template <typename R, typename OutT>
__device__ __forceinline__ void xfer_write(const Camera &c, const R C[4], int ix, int iy, XChain<R> &Ln, void *out,
                                           void *depth) {
#pragma unroll
    for (int i = 0; i < 4; i++) Ln.S[i] += Ln.Slo[i];
    reproject(C, Ln.S);
    long long pix = (long long)iy * c.nx + ix;
    OutT *o = reinterpret_cast<OutT *>(out) + 4 * pix;
    o[0] = OutT(Ln.S[0]);
    o[1] = OutT(Ln.S[1]);
    o[2] = OutT(Ln.S[2]);
    o[3] = OutT(Ln.S[3]);
    if (depth) {
        OutT *d = reinterpret_cast<OutT *>(depth) + 2 * pix;
        d[0] = OutT(Ln.tau - Ln.tauc);
        d[1] = OutT(Ln.phi - Ln.phic);
    }
}

template <typename R, typename OutT>
__device__ __forceinline__ void xfer_finish(const Camera &c, const KS<R> &m, int ix, int iy, XLane<R> &Ln, void *out,
                                            void *depth) {
    R C[4];
    camera_matrix<R>(c, m, ix, iy, Ln, C);
    xfer_write<R, OutT>(c, C, ix, iy, Ln, out, depth);
}

// A pixel whose ray has no usable path: zero Stokes (and depths).
template <typename OutT>
__device__ __forceinline__ void xfer_zero(long long pix, void *out, void *depth) {
    OutT *o = reinterpret_cast<OutT *>(out) + 4 * pix;
    o[0] = o[1] = o[2] = o[3] = OutT(0);
    if (depth) {
        OutT *d = reinterpret_cast<OutT *>(depth) + 2 * pix;
        d[0] = d[1] = OutT(0);
    }
}

// What the thermal coefficients read: in FP32 the Bessel quadrature's weights exp(-(k h)^2) (halved at
// k = 0), put into shared memory here, in FP64 the tables in global memory.
__device__ __forceinline__ const float *thermal_weights(float *sgw, const double *) {
    if (threadIdx.x < BesselCfg::nq) {
        float u = float(threadIdx.x) * BesselCfg::h;
        sgw[threadIdx.x] = expf(-u * u) * (threadIdx.x == 0 ? 0.5f : 1.0f);
    }
    return sgw;
}
__device__ __forceinline__ const double *thermal_weights(double *, const double *tab) { return tab; }

// JOBS: the rays run over a table of images (p.jobs), each with its own camera, model and
// outputs; otherwise over the one image of p.cam, p.model, p.out.
template <typename R, typename OutT, int CM = 0, bool JOBS = false>
__global__ void __launch_bounds__(kXferThreads, sizeof(R) == 4 ? 4 : 1) transfer_kernel(XferArgs p) {
    if (sizeof(R) == 8 && p.records && record_tail(p)) return;  // the two kernels have run
    __shared__ R wsh[sizeof(R) == 4 ? 32 : 1];
    const R *sgw = thermal_weights(wsh, p.therm);
    __syncthreads();
    long long ray = -1;
    int blk = -1, slot = 0, n = 0, rstat = 0, job = 0;
    bool live = false, drained = false;
    XLane<R> Ln;
    unsigned long long my_pts = 0, my_emit = 0;
    // this ray's image: pixel, and (JOBS) the job's camera, model and outputs
    auto gid_of = [&](long long r) { return p.pix_list ? (long long)p.pix_list[r + p.ray_offset] : r + p.ray_offset; };
    auto pixel = [&](int &ix, int &iy) {
        if (JOBS) {
            const JobDev &J = p.jobs[job];
            ray_pixel(gid_of(ray) - J.ray_begin, J.cam.nx, J.cam.ny, ix, iy);
        } else {
            map_pixel(p.pix_list, ray + p.ray_offset, p.cam.nx, p.cam.ny, ix, iy);
        }
    };
    for (;;) {
        bool want = !live && !drained;
        unsigned long long t = warp_pop(&p.ctr->xfer_next, want);
        if (want) {
            if (t < (unsigned long long)p.nrays) {
                ray = (long long)t;
                if (JOBS) job = find_job(p.jobs, p.njobs, gid_of(ray));
                RayRecord rec = p.rec[ray];
                rstat = rec.status;
                if (rec.nstates >= 2) {
                    blk = rec.last_block;
                    slot = (rec.nstates - 1) % kBlockStates;
                    n = rec.nstates - 1;
                    Ln.reset();
                    live = true;
                } else {
                    int ix, iy;
                    pixel(ix, iy);
                    const Camera &c = JOBS ? p.jobs[job].cam : p.cam;
                    void *out = JOBS ? p.jobs[job].out : p.out, *depth = JOBS ? p.jobs[job].depth : p.depth;
                    uint8_t *status = JOBS ? p.jobs[job].status : p.status;
                    long long pix = (long long)iy * c.nx + ix;
                    xfer_zero<OutT>(pix, out, depth);
                    if (status) status[pix] = (uint8_t)rstat;
                }
            } else {
                drained = true;
            }
        }
        if (__all_sync(0xffffffffu, !live && drained)) break;
        if (!live) continue;

        // move from state n to state n-1
        if (--slot < 0) {
            blk = p.arena.prev[blk];
            slot = kBlockStates - 1;
        }
        n--;
        const double4_32a *src = reinterpret_cast<const double4_32a *>(p.arena.states + (long long)blk * kBlockStates + slot);
        double4_32a q0 = src[0], q1 = src[1];
        KS<R> m;
        const Camera &c = JOBS ? p.jobs[job].cam : p.cam;
        const Model &mdl = JOBS ? p.jobs[job].model : p.model;
        if (xfer_point<R, CM>(c, mdl, q0, q1, sgw, Ln, m, &p, (long long)blk * kBlockStates + slot)) my_emit++;
        my_pts++;
        if (n == 0) {
            int ix, iy;
            pixel(ix, iy);
            void *out = JOBS ? p.jobs[job].out : p.out, *depth = JOBS ? p.jobs[job].depth : p.depth;
            uint8_t *status = JOBS ? p.jobs[job].status : p.status;
            xfer_finish<R, OutT>(c, m, ix, iy, Ln, out, depth);
            if (status) status[(long long)iy * c.nx + ix] = (uint8_t)rstat;
            live = false;
        }
    }
    if (my_pts) atomicAdd(&p.ctr->points, my_pts);
    if (my_emit) atomicAdd(&p.ctr->emitting, my_emit);
}

// ---- The transfer as two kernels -------------------------------------------------------------
// A state's record, in place of the state (64 bytes: in FP32 the 12 values, in FP64 the first 8,
// the other 4 at tail), and a ray's camera matrix in place of its last state, which no step leaves.
template <typename R>
__device__ __forceinline__ void store_rec(const XferArgs &p, double *tail, long long st, const XRec<R> &x) {
    if constexpr (sizeof(R) == 4) {
        float4 *d = reinterpret_cast<float4 *>(p.arena.states + st);
        d[0] = make_float4(x.d11, x.d12, x.d21, x.d22);
        d[1] = make_float4(x.tau, x.aQ, x.aV, x.rQ);
        d[2] = make_float4(x.rV, x.J0, x.J1, x.J3);
    } else {
        double4_32a *d = reinterpret_cast<double4_32a *>(p.arena.states + st);
        d[0] = make_double4_32a(x.d11, x.d12, x.d21, x.d22);
        d[1] = make_double4_32a(x.tau, x.aQ, x.aV, x.rQ);
        reinterpret_cast<double4_32a *>(tail)[st] = make_double4_32a(x.rV, x.J0, x.J1, x.J3);
    }
}
template <typename R>
__device__ __forceinline__ XRec<R> load_rec(const XferArgs &p, const double *tail, long long st) {
    if constexpr (sizeof(R) == 4) {
        const float4 *d = reinterpret_cast<const float4 *>(p.arena.states + st);
        const float4 a = d[0], b = d[1], c = d[2];
        return XRec<R>{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w};
    } else {
        const double4_32a *d = reinterpret_cast<const double4_32a *>(p.arena.states + st);
        const double4_32a a = d[0], b = d[1], c = reinterpret_cast<const double4_32a *>(tail)[st];
        return XRec<R>{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w};
    }
}

template <typename R>
__device__ __forceinline__ void shfl_legs(const XLegs<R> &L, const XLegs<R> &carry, int lane, XLegs<R> &in) {
    const unsigned full = 0xffffffffu;
    const bool top = lane == 31;
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const R a = __shfl_down_sync(full, L.eo1[i], 1), b = __shfl_down_sync(full, L.eo2[i], 1);
        const R c = __shfl_down_sync(full, L.u1[i], 1), d = __shfl_down_sync(full, L.u2[i], 1);
        const R e = __shfl_down_sync(full, L.a1[i], 1), f = __shfl_down_sync(full, L.a2[i], 1);
        in.eo1[i] = top ? carry.eo1[i] : a, in.eo2[i] = top ? carry.eo2[i] : b;
        in.u1[i] = top ? carry.u1[i] : c, in.u2[i] = top ? carry.u2[i] : d;
        in.a1[i] = top ? carry.a1[i] : e, in.a2[i] = top ? carry.a2[i] : f;
    }
    const int b = __shfl_down_sync(full, (int)L.basis, 1);
    in.basis = top ? carry.basis : b != 0;
}
template <typename R>
__device__ __forceinline__ void first_lane_legs(const XLegs<R> &L, XLegs<R> &carry) {
    const unsigned full = 0xffffffffu;
#pragma unroll
    for (int i = 0; i < 4; i++) {
        carry.eo1[i] = __shfl_sync(full, L.eo1[i], 0), carry.eo2[i] = __shfl_sync(full, L.eo2[i], 0);
        carry.u1[i] = __shfl_sync(full, L.u1[i], 0), carry.u2[i] = __shfl_sync(full, L.u2[i], 0);
        carry.a1[i] = __shfl_sync(full, L.a1[i], 0), carry.a2[i] = __shfl_sync(full, L.a2[i], 0);
    }
    carry.basis = __shfl_sync(full, (int)L.basis, 0) != 0;
}

template <typename R>
struct PointsCfg;
// FP32: about 2,700 instructions per 32 states in a straight line, more than the instruction cache
// holds: with every warp at its own place in it, waiting for instructions is the largest stall. A
// barrier per 32 states keeps a block's warps together (1024^2 torus, points and chain: 128 threads
// without it 69.9 ms, 256 threads with it 63.5, 512 63.1), and 3 blocks of 256 at 84 registers beat
// 2 at 128 (61.2 ms).
template <>
struct PointsCfg<float> {
    static constexpr int threads = 256, blocks = 3;
    static constexpr bool sync = true;
};
template <>
struct PointsCfg<double> {
    static constexpr int threads = 128, blocks = 1;
    static constexpr bool sync = false;
};

// The geometry of every saved state: one warp per ray, one lane per state of an arena block, from
// the ray's last block to its first. A lane's step needs the legs that leave its far neighbour: the
// next lane's, or for the block's last state those of the block before (carry). Where a state emits
// they are its own fluid screen, at once; legs that pass through states that do not emit are
// handed down lane by lane, which is dearer than a state that emits: a torus on a grid of 50 M seen from
// 1000 M (47% of the states outside it) takes 84.5 ms of transfer at 1024^2 (91.6 when also the states
// beyond the first emission were handed nothing, lane by lane), with every state emitting 61.0; the one-lane
// kernel took 65.4 and 69.0.
template <typename R, int CM = 0, bool JOBS = false>
__global__ void __launch_bounds__(PointsCfg<R>::threads, PointsCfg<R>::blocks) points_kernel(XferArgs p) {
    double *const tail = sizeof(R) == 8 ? record_tail(p) : nullptr;
    if (sizeof(R) == 8 && !tail) return;
    __shared__ R wsh[sizeof(R) == 4 ? 32 : 1];
    const R *sgw = thermal_weights(wsh, p.therm);
    __syncthreads();
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    unsigned long long my_pts = 0, my_emit = 0;
    const JobDev *J = nullptr;
    long long ray = 0, gid = 0, last = 0;
    int N = 0, base = -1, blk = -1;  // the ray's states that a step leaves, and the next block's first state
    bool drained = false;
    XLegs<R> carry;
    for (;;) {
        if (base < 0 && !drained) {
            unsigned long long t = 0;
            if (lane == 0) t = atomicAdd(&p.ctr->xfer_next, 1ull);
            t = __shfl_sync(full, t, 0);
            drained = t >= (unsigned long long)p.nrays;
            if (!drained) {
                ray = (long long)t;
                const RayRecord rec = p.rec[ray];
                if (rec.nstates >= 2) {
                    gid = p.pix_list ? (long long)p.pix_list[ray + p.ray_offset] : ray + p.ray_offset;
                    if (JOBS) J = p.jobs + find_job(p.jobs, p.njobs, gid);
                    N = rec.nstates - 1;
                    blk = rec.last_block;
                    last = (long long)blk * kBlockStates + N % kBlockStates;
                    base = N / kBlockStates * kBlockStates;
                    if (base == N) {  // the last block holds the last state alone
                        base -= kBlockStates;
                        blk = p.arena.prev[blk];
                    }
#pragma unroll
                    for (int i = 0; i < 4; i++)
                        carry.eo1[i] = carry.eo2[i] = carry.u1[i] = carry.u2[i] = carry.a1[i] = carry.a2[i] = R(0);
                    carry.basis = false;
                }
            }
        }
        if (PointsCfg<R>::sync ? __syncthreads_and(drained) : drained) break;
        if (base < 0) continue;
        const Camera &c = JOBS ? J->cam : p.cam;
        const Model &mdl = JOBS ? J->model : p.model;
        const int prev = base > 0 ? p.arena.prev[blk] : -1;
        const bool act = base + lane < N;
        const long long st = (long long)blk * kBlockStates + lane;
        XPoint<R> P;
        XRec<R> x;
        XLegs<R> L;
        R T0[4][4];
        P.valid = false;
        L.basis = false;
#pragma unroll
        for (int i = 0; i < 4; i++) L.eo1[i] = L.eo2[i] = L.u1[i] = L.u2[i] = L.a1[i] = L.a2[i] = R(0);
        if (act) {
            const double4_32a *src = reinterpret_cast<const double4_32a *>(p.arena.states + st);
            const double4_32a q0 = src[0], q1 = src[1];
            xfer_eval<R, CM>(c, mdl, q0, q1, sgw, P, x, &p, st);
            connection_T(P.m, P.K, T0);
            if (P.valid) xfer_screen(P, T0, L);
        }
        // nothing comes down to the states beyond which none emits
        const unsigned emit = __ballot_sync(full, P.valid);
        bool done = P.valid || !act || (!carry.basis && emit >> lane == 0u);
        XLegs<R> in;
        unsigned mask = __ballot_sync(full, done);
        while (mask != full) {
            shfl_legs(L, carry, lane, in);
            if (!done && (lane == 31 || ((mask >> (lane + 1)) & 1u))) {
                L = in;
                if (in.basis) {
                    xfer_link(P, T0, L, x);
                    xfer_pass(T0, L);
                }
                done = true;
            }
            mask = __ballot_sync(full, done);
        }
        shfl_legs(L, carry, lane, in);
        if (act) {
            if (P.valid)
                xfer_link(P, T0, in, x);
            else
                x.tau = R(-INFINITY);
            store_rec(p, tail, st, x);
        }
        if (base == 0 && lane == 0) {
            int ix, iy;
            if (JOBS)
                ray_pixel(gid - J->ray_begin, c.nx, c.ny, ix, iy);
            else
                map_pixel(p.pix_list, ray + p.ray_offset, c.nx, c.ny, ix, iy);
            R C[4];
            camera_matrix<R>(c, P.m, ix, iy, L, C);
            R *d = reinterpret_cast<R *>(p.arena.states + last);
#pragma unroll
            for (int i = 0; i < 4; i++) d[i] = C[i];
        }
        first_lane_legs(L, carry);
        my_pts += act;
        my_emit += act && P.valid;
        blk = prev;
        base -= kBlockStates;
    }
    if (my_pts) atomicAdd(&p.ctr->points, my_pts);
    if (my_emit) atomicAdd(&p.ctr->emitting, my_emit);
}

// The Stokes chain: one lane per ray (per-lane refill from a queue), from the far end to the camera
// over the records of points_kernel; the next record is loaded before the current one is applied.
template <typename R, typename OutT, bool JOBS = false>
__global__ void __launch_bounds__(kXferThreads) chain_kernel(XferArgs p) {
    const double *const tail = sizeof(R) == 8 ? record_tail(p) : nullptr;
    if (sizeof(R) == 8 && !tail) return;
    long long ray = -1;
    int blk = -1, slot = 0, n = 0, rstat = 0, job = 0;
    bool live = false, drained = false;
    XChain<R> Ln;
    XRec<R> next;
    R C[4];
    auto gid_of = [&](long long r) { return p.pix_list ? (long long)p.pix_list[r + p.ray_offset] : r + p.ray_offset; };
    auto pixel = [&](int &ix, int &iy) {
        if (JOBS) {
            const JobDev &J = p.jobs[job];
            ray_pixel(gid_of(ray) - J.ray_begin, J.cam.nx, J.cam.ny, ix, iy);
        } else {
            map_pixel(p.pix_list, ray + p.ray_offset, p.cam.nx, p.cam.ny, ix, iy);
        }
    };
    auto step_back = [&]() {
        if (--slot < 0) {
            blk = p.arena.prev[blk];
            slot = kBlockStates - 1;
        }
        next = load_rec<R>(p, tail, (long long)blk * kBlockStates + slot);
    };
    for (;;) {
        bool want = !live && !drained;
        unsigned long long t = warp_pop(&p.ctr->chain_next, want);
        if (want) {
            if (t < (unsigned long long)p.nrays) {
                ray = (long long)t;
                if (JOBS) job = find_job(p.jobs, p.njobs, gid_of(ray));
                RayRecord rec = p.rec[ray];
                rstat = rec.status;
                if (rec.nstates >= 2) {
                    blk = rec.last_block;
                    slot = (rec.nstates - 1) % kBlockStates;
                    n = rec.nstates - 1;
                    const R *d = reinterpret_cast<const R *>(p.arena.states + (long long)blk * kBlockStates + slot);
#pragma unroll
                    for (int i = 0; i < 4; i++) C[i] = d[i];
                    Ln.reset();
                    step_back();
                    live = true;
                } else {
                    int ix, iy;
                    pixel(ix, iy);
                    const Camera &c = JOBS ? p.jobs[job].cam : p.cam;
                    void *out = JOBS ? p.jobs[job].out : p.out, *depth = JOBS ? p.jobs[job].depth : p.depth;
                    uint8_t *status = JOBS ? p.jobs[job].status : p.status;
                    long long pix = (long long)iy * c.nx + ix;
                    xfer_zero<OutT>(pix, out, depth);
                    if (status) status[pix] = (uint8_t)rstat;
                }
            } else {
                drained = true;
            }
        }
        if (__all_sync(0xffffffffu, !live && drained)) break;
        if (!live) continue;
        n--;
        const XRec<R> x = next;
        if (n > 0) step_back();
        if (!(x.tau == R(-INFINITY))) Ln.apply(x);
        if (n == 0) {
            int ix, iy;
            pixel(ix, iy);
            const Camera &c = JOBS ? p.jobs[job].cam : p.cam;
            void *out = JOBS ? p.jobs[job].out : p.out, *depth = JOBS ? p.jobs[job].depth : p.depth;
            uint8_t *status = JOBS ? p.jobs[job].status : p.status;
            xfer_write<R, OutT>(c, C, ix, iy, Ln, out, depth);
            if (status) status[(long long)iy * c.nx + ix] = (uint8_t)rstat;
            live = false;
        }
    }
}

// ---- The grid fetch staged through shared memory by TMA (FP32 form, thermal electrons) ----
// Each lane owns a 256-byte slot of shared memory and an mbarrier. While it works on one saved
// state, the 2 x 2 x 2 cells of the next state's trilinear stencil are copied into its slot by
// one TMA tensor load: a box of 8 floats x 2 x 2 x 2 cells of the grid seen as a 4-d tensor
// [n1][n2][n3][8]. The fetch's latency then hides behind a whole point of work, and the eight
// 32-byte gathers leave the load/store path. At the periodic seam in phi (k1 = 0) the two
// k cells are not adjacent in memory, and the lane copies that stencil with plain loads. The
// interpolation takes the cells in grid_interp's order, so the image is the same bit for bit.

// TMA: the box of the 4-d tensor map at coordinates (c0, c1, c2, c3), innermost first, into
// shared memory at dst, counted on the mbarrier bar's transaction bytes.
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, int c3,
                                            uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];\n" ::"r"(dst),
        "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
        : "memory");
}

// Arrive on bar (this thread's one arrival) and expect bytes more of transactions.
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}

// The staged cells of one state in grid_interp's order: cell (di, dj, dk) at float4
// ((di 2 + dj) 2 + dk) 2 (and + 1).
template <typename R>
__device__ __forceinline__ void grid_interp_staged(const GridCell<R> &c, const float4 *s, R P[8]) {
#pragma unroll
    for (int q = 0; q < 8; q++) P[q] = R(0);
#pragma unroll
    for (int di = 0; di < 2; di++)
#pragma unroll
        for (int dj = 0; dj < 2; dj++) {
            R wij = (di ? c.w1 : R(1) - c.w1) * (dj ? c.w2 : R(1) - c.w2);
#pragma unroll
            for (int dk = 0; dk < 2; dk++) {
                R wt = wij * (dk ? c.w3 : R(1) - c.w3);
                const int o = ((di * 2 + dj) * 2 + dk) * 2;
                float4 lo = s[o], hi = s[o + 1];
                P[0] += wt * R(lo.x);
                P[1] += wt * R(lo.y);
                P[2] += wt * R(lo.z);
                P[3] += wt * R(lo.w);
                P[4] += wt * R(hi.x);
                P[5] += wt * R(hi.y);
                P[6] += wt * R(hi.z);
                P[7] += wt * R(hi.w);
            }
        }
}

// CM: the coefficients (0: thermal fits; the only one staged so far)
template <int CM = 0>
__global__ void __launch_bounds__(kXferThreads, 4) transfer_kernel_staged(XferArgs p, const __grid_constant__ CUtensorMap tmap) {
    typedef float R;
    __shared__ R sgw[32];
    __shared__ __align__(128) float4 stc[kXferThreads * 16];
    __shared__ __align__(8) unsigned long long bars[kXferThreads];
    thermal_weights(sgw, p.therm);
    const uint32_t bar = smem_u32(&bars[threadIdx.x]);
    float4 *slot_s = stc + threadIdx.x * 16;
    const uint32_t slot_a = smem_u32(slot_s);
    mbar_init(bar, 1);
    __syncthreads();
    const GridModel &g = p.model.grid;
    long long ray = -1;
    int blk = -1, slot = 0, n = 0, rstat = 0;
    bool live = false, drained = false, failed = false;
    XLane<R> Ln;
    unsigned long long my_pts = 0, my_emit = 0;
    uint32_t phase = 0;
    // the next state's cell, and where its stencil is: 0 nowhere (outside the grid), 1 in
    // flight (TMA), 2 in the slot (plain loads at the seam)
    GridCell<R> nc;
    int nmode = 0;
    auto stage = [&](int b, int s) {
        const double4_32a q = *reinterpret_cast<const double4_32a *>(p.arena.states + (long long)b * kBlockStates + s);
        nmode = 0;
        if (!grid_cell<R>(g, q.x, q.y, q.z, nc)) return;
        if (nc.k1 != 0) {
            fence_smem_async();  // the slot's last reads (generic proxy) before the TMA's writes
            mbar_expect_tx(bar, 16 * sizeof(float4));
            tma_load_4d(slot_a, &tmap, 0, nc.k0, nc.j0, nc.i0, bar);
            nmode = 1;
        } else {
#pragma unroll
            for (int di = 0; di < 2; di++)
#pragma unroll
                for (int dj = 0; dj < 2; dj++) {
                    long long row = ((long long)(nc.i0 + di) * g.n2 + (nc.j0 + dj)) * g.n3;
#pragma unroll
                    for (int dk = 0; dk < 2; dk++) {
                        long long cell = row + (dk ? nc.k1 : nc.k0);
                        const int o = ((di * 2 + dj) * 2 + dk) * 2;
                        slot_s[o] = __ldg(g.prims + 2 * cell);
                        slot_s[o + 1] = __ldg(g.prims + 2 * cell + 1);
                    }
                }
            nmode = 2;
        }
    };
    // the state after (b, s) on the walk toward the camera
    auto step_back = [&](int &b, int &s) {
        if (--s < 0) {
            b = p.arena.prev[b];
            s = kBlockStates - 1;
        }
    };
    for (;;) {
        bool want = !live && !drained;
        unsigned long long t = warp_pop(&p.ctr->xfer_next, want);
        if (want) {
            if (t < (unsigned long long)p.nrays) {
                ray = (long long)t;
                RayRecord rec = p.rec[ray];
                rstat = rec.status;
                if (rec.nstates >= 2) {
                    blk = rec.last_block;
                    slot = (rec.nstates - 1) % kBlockStates;
                    n = rec.nstates - 1;
                    Ln.reset();
                    live = true;
                    int b1 = blk, s1 = slot;
                    step_back(b1, s1);
                    stage(b1, s1);
                } else {
                    int ix, iy;
                    map_pixel(p.pix_list, ray + p.ray_offset, p.cam.nx, p.cam.ny, ix, iy);
                    long long pix = (long long)iy * p.cam.nx + ix;
                    xfer_zero<R>(pix, p.out, p.depth);
                    if (p.status) p.status[pix] = (uint8_t)rstat;
                }
            } else {
                drained = true;
            }
        }
        if (__all_sync(0xffffffffu, !live && drained)) break;
        if (!live) continue;

        step_back(blk, slot);
        n--;
        const double4_32a *src = reinterpret_cast<const double4_32a *>(p.arena.states + (long long)blk * kBlockStates + slot);
        double4_32a q0 = src[0], q1 = src[1];
        // this state's primitives from the slot, then the next state's stencil into it
        const GridCell<R> cc = nc;
        const int cmode = nmode;
        R P[8];
        if (cmode == 1 && !failed) {
            if (mbar_wait(bar, phase))
                phase ^= 1u;
            else
                failed = true;  // the copy is still owed on this phase
        }
        if (cmode != 0) grid_interp_staged(cc, slot_s, P);
        if (n > 0 && !failed) {
            int b1 = blk, s1 = slot;
            step_back(b1, s1);
            stage(b1, s1);
        } else {
            nmode = 0;
        }
        KS<R> m;
        PreFetch<R> pre{cmode != 0 && !failed ? &cc : nullptr, P};
        if (xfer_point<R, CM, true>(p.cam, p.model, q0, q1, sgw, Ln, m, &p, 0, pre)) my_emit++;
        my_pts++;
        if (n == 0) {
            int ix, iy;
            map_pixel(p.pix_list, ray + p.ray_offset, p.cam.nx, p.cam.ny, ix, iy);
            xfer_finish<R, R>(p.cam, m, ix, iy, Ln, p.out, p.depth);
            if (p.status) p.status[(long long)iy * p.cam.nx + ix] = (uint8_t)rstat;
            live = false;
        }
    }
    if (failed) {  // report, and give the copy in flight (bounded) time to land before exit
        atomicAdd(&p.ctr->n_status[kStageStatus], 1u);
        mbar_wait(bar, phase);
    }
    if (my_pts) atomicAdd(&p.ctr->points, my_pts);
    if (my_emit) atomicAdd(&p.ctr->emitting, my_emit);
}

// The surrogate form's features pass: for every emitting saved state the network's normalised inputs
// (f mapped from the box to [-1, 1]); other states get zeros. Same arithmetic as the transfer's own
// feature evaluation. One warp per ray, one lane per state of an arena block (as points_kernel).
template <typename R>
__global__ void __launch_bounds__(kXferThreads, 5) sur_features_pass(XferArgs p) {
    const Camera &c = p.cam;
    const R a = pick<R>(c.a, c.f_a), nu_obs = pick<R>(c.nu_obs, c.f_nu_obs);
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    long long row = 0;
    int N = 0, base = -1, blk = -1;  // as in points_kernel
    for (;;) {
        if (base < 0) {
            unsigned long long t = 0;
            if (lane == 0) t = atomicAdd(&p.ctr->feat_next, 1ull);
            t = __shfl_sync(full, t, 0);
            if (t >= (unsigned long long)p.nrays) break;
            const RayRecord rec = p.rec[t];
            if (rec.nstates < 2) continue;
            N = rec.nstates - 1;
            blk = rec.last_block;
            base = N / kBlockStates * kBlockStates;
            if (base == N) {  // the last block holds the last state alone
                base -= kBlockStates;
                blk = p.arena.prev[blk];
            }
            // compact rows: the ray's N states take N consecutive rows
            if (p.sur_row) {
                if (lane == 0) row = (long long)atomicAdd(&p.ctr->sur_rows, (unsigned long long)N);
                row = __shfl_sync(full, row, 0);
            }
        }
        const int prev = base > 0 ? p.arena.prev[blk] : -1;
        const bool act = base + lane < N;
        const long long st = (long long)blk * kBlockStates + lane;
        bool valid = false;
        float f[4];
        if (act) {
            const double4_32a *src = reinterpret_cast<const double4_32a *>(p.arena.states + st);
            const double4_32a q0 = src[0], q1 = src[1];
            R r = to_real<R>(q0.x), th = to_real<R>(q0.y);
            R K[4] = {to_real<R>(q0.w), to_real<R>(q1.x), to_real<R>(q1.y), to_real<R>(q1.z)};
            KS<R> m;
            m.eval(a, r, th);
            Plasma<R> pl;
            if (p.model.kind == 1)
                adaf_plasma(p.model.adaf, a, m, r, pl);
            else
                grid_plasma(p.model.grid, m, q0.x, q0.y, q0.z, pl);
            float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
            valid = pl.valid;
            if (valid) {
                R e1[4], e2[4], w, sth, cth;
                fluid_tetrad(m, K, pl.u, pl.b, e1, e2, w, sth, cth);
                float xn[4];
                sur_features_r<R>(pl.Te, pl.B, w * nu_obs, sth, cth, R(p.model.kappa), f);
#pragma unroll
                for (int j = 0; j < 4; j++) xn[j] = 2.0f * (f[j] - p.sur_lo[j]) / (p.sur_hi[j] - p.sur_lo[j]) - 1.0f;
                o = make_float4(xn[0], xn[1], xn[2], xn[3]);
            }
            if (p.sur_row) {
                p.feat[row + base + lane] = o;
                p.sur_row[st] = (int)(row + base + lane);
            } else if (p.feat) {
                p.feat[st] = o;
            }
        }
        if (p.feat_raw) {  // one counter update a warp
            const unsigned em = __ballot_sync(full, valid);
            unsigned long long k = 0;
            if (lane == 0 && em) k = atomicAdd(&p.ctr->feat_count, (unsigned long long)__popc(em));
            k = __shfl_sync(full, k, 0) + __popc(em & ((1u << lane) - 1u));
            if (valid && (long long)k < p.feat_cap) p.feat_raw[k] = make_float4(f[0], f[1], f[2], f[3]);
        }
        blk = prev;
        base -= kBlockStates;
    }
}

// The unpolarized transfer (Stokes I only, for fitting loops): I/nu^3 is a scalar invariant,
// so nothing is transported. At each emitting point: the pitch angle from scalar products
// (the ray's fluid-frame direction is -K - w u, b is spatial in that frame), j_I and a_I, and the
// exact step I <- I e^-tau + (j ds / w^3) (1 - e^-tau)/tau, added as the increment
// (J - tau I) (1 - e^-tau)/tau with TwoSum compensation. Output: one value per pixel.
// One warp per ray, one lane per state of an arena block (as points_kernel); the increments of the
// block's emitting states then follow one another, every lane adding the value that the state's lane
// holds (11 instructions a state). With one lane per ray the states of a ray were a serial chain of a
// point's whole evaluation each, and 16,384 rays filled a ninth of the chip: a torus at 128^2 took
// 7.1 ms, now 0.78, at 1024^2 34.8 (256 threads and 3 blocks, with or without a barrier per block of
// states, 34.7 and 36.0; 128 threads and 4 blocks 39.8).
template <typename R, bool JOBS = false>
__global__ void __launch_bounds__(kXferThreads, 6) unpol_kernel(XferArgs p) {
    typedef Mth<R> F;
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    unsigned long long my_pts = 0, my_emit = 0;
    const JobDev *J = nullptr;
    long long ray = 0, gid = 0;
    int N = 0, base = -1, blk = -1, rstat = 0;  // as in points_kernel
    bool drained = false;
    R I = 0, Ilo = 0;
    for (;;) {
        if (base < 0 && !drained) {
            unsigned long long t = 0;
            if (lane == 0) t = atomicAdd(&p.ctr->xfer_next, 1ull);
            t = __shfl_sync(full, t, 0);
            drained = t >= (unsigned long long)p.nrays;
            if (!drained) {
                ray = (long long)t;
                const RayRecord rec = p.rec[ray];
                gid = p.pix_list ? (long long)p.pix_list[ray + p.ray_offset] : ray + p.ray_offset;
                if (JOBS) J = p.jobs + find_job(p.jobs, p.njobs, gid);
                rstat = rec.status;
                N = max(rec.nstates - 1, 0);
                blk = rec.last_block;
                base = N / kBlockStates * kBlockStates;
                if (base == N && N > 0) {  // the last block holds the last state alone
                    base -= kBlockStates;
                    blk = p.arena.prev[blk];
                }
                I = Ilo = R(0);
            }
        }
        if (drained) break;
        if (base < 0) continue;
        const Camera &c = JOBS ? J->cam : p.cam;
        const int prev = base > 0 ? p.arena.prev[blk] : -1;
        bool valid = false;
        R tau = 0, Jn = 0, ph1 = 0;
        if (base + lane < N) {
            const double4_32a *src = reinterpret_cast<const double4_32a *>(p.arena.states + (long long)blk * kBlockStates + lane);
            const double4_32a q0 = src[0], q1 = src[1];
            R r = to_real<R>(q0.x), th = to_real<R>(q0.y);
            R K[4] = {to_real<R>(q0.w), to_real<R>(q1.x), to_real<R>(q1.y), to_real<R>(q1.z)};
            R h = fabs(to_real<R>(q1.w));
            KS<R> m;
            m.eval(pick<R>(c.a, c.f_a), r, th);
            Plasma<R> pl;
            const Model &mdl = JOBS ? J->model : p.model;
            if (mdl.kind == 1)
                adaf_plasma(mdl.adaf, pick<R>(c.a, c.f_a), m, r, pl);
            else
                grid_plasma(mdl.grid, m, q0.x, q0.y, q0.z, pl);
            valid = pl.valid;
            if (valid) {
                R w = m.dot(K, pl.u);
                R kp[4], bn[4];
                R bs = fmax(fmax(fabs(pl.b[0]), fabs(pl.b[1])), fmax(fabs(pl.b[2]), fabs(pl.b[3])));
                R ibs = bs > R(0) ? R(1) / bs : R(0);
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    kp[i] = -K[i] - w * pl.u[i];
                    bn[i] = pl.b[i] * ibs;
                }
                R bb = m.dot(bn, bn), kk = m.dot(kp, kp), bk = m.dot(bn, kp);
                R sth = (bb > R(0) && kk > R(0)) ? F::sqrt_(fmax(bb - bk * bk / kk, R(0)) / bb) : R(0);
                R jI, aI;
                thermal_jI_aI(pl.ne, pl.Te, pl.B, w * pick<R>(c.nu_obs, c.f_nu_obs), sth, jI, aI);
                R ds = w * h * pick<R>(c.L_unit, c.f_L_unit);
                tau = aI * ds;
                Jn = jI * ds / (w * w * w);
                ph1 = phi1(tau);
            }
            my_pts++;
            my_emit += valid;
        }
        for (unsigned em = __ballot_sync(full, valid); em;) {
            const int j = 31 - __clz(em);
            em ^= 1u << j;
            const R tj = __shfl_sync(full, tau, j), Jj = __shfl_sync(full, Jn, j), pj = __shfl_sync(full, ph1, j);
            two_sum_add(I, Ilo, (Jj - tj * I) * pj);
        }
        if (base == 0 && lane == 0) {
            int ix, iy;
            if (JOBS)
                ray_pixel(gid - J->ray_begin, c.nx, c.ny, ix, iy);
            else
                map_pixel(p.pix_list, ray + p.ray_offset, c.nx, c.ny, ix, iy);
            const long long pix = (long long)iy * c.nx + ix;
            reinterpret_cast<R *>(JOBS ? J->out : p.out)[pix] = N > 0 ? I + Ilo : R(0);
            uint8_t *status = JOBS ? J->status : p.status;
            if (status) status[pix] = (uint8_t)rstat;
        }
        blk = prev;
        base -= kBlockStates;
    }
    if (my_pts) atomicAdd(&p.ctr->points, my_pts);
    if (my_emit) atomicAdd(&p.ctr->emitting, my_emit);
}

}  // namespace prt
