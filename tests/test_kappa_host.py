"""The kappa quadrature (csrc/kappa.cuh), compiled for the CPU with tables built as the library builds them,
against the same integrals in long double by the trapezoid rule from far below to far above every
scale of the integrands. Tolerances: 2e-9 relative for emission and absorption (4e-10 from the nodes
and the light-cone scaling of Q and V by a ratio of two of them), to which absorption adds the rounding of
the terms it is a difference of, about 1 / (Theta_e X) times itself for cold electrons; 1e-13 for the
rotativities (a few hundred terms of one sign, each rounded a few times). No GPU is used."""
import ctypes
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

import __graft_entry__  # noqa: F401  (puts the repo root on sys.path)

E, ME, C = 4.80320471257e-10, 9.1093837015e-28, 2.99792458e10

SRC = r"""
#include <algorithm>
#include <cmath>
#include <vector>
#define __device__
#define __forceinline__ inline
using std::max;
using std::min;
static double rsqrt(double x) { return 1.0 / std::sqrt(x); }
typedef long double L;
static const L PI = 3.14159265358979323846264338327950288L;
static double chebyshev(int j, int n) { return (double)cosl(PI * j * (n + 0.5L) / 8); }
namespace prt {
constexpr double kC = 2.99792458e10, kMe = 9.1093837015e-28, kQe = 4.80320471257e-10, kPi = 3.14159265358979323846;
struct KapNode;
struct KappaTables { const double *kern; const KapNode *node; };
}
#include "kappa_host.h"
using namespace prt;
static std::vector<double> kern(24 * kSynN);
static std::vector<KapNode> node(kKapN);
extern "C" void tables() {
    for (int k = 0; k < kKapN; k++) node[k] = kap_node(kKapLo + k * kKapH);
    for (int i = 0; i < kSynN; i++) {
        double f[3][8];
        for (int j = 0; j < 8; j++) {
            const double lx = kSynLo + (i + 0.5 + 0.5 * chebyshev(1, j)) * 0.125;
            double k[3];
            synch_kernels_scaled(exp(lx), k);
            for (int m = 0; m < 3; m++) f[m][j] = k[m] * exp(-lx * (1.0 / 3.0));
        }
        for (int m = 0; m < 3; m++) {
            double p[8] = {0}, a[8] = {1}, b[8] = {0, 1};
            for (int n = 0; n < 8; n++) {
                double s = 0.0, c[8];
                for (int j = 0; j < 8; j++) s += f[m][j] * chebyshev(n, j);
                for (int q = 0; q < 8; q++) {
                    p[q] += s * (n ? 0.25 : 0.125) * a[q];
                    c[q] = (q ? 2.0 * b[q - 1] : 0.0) - a[q];
                }
                for (int q = 0; q < 8; q++) a[q] = b[q], b[q] = c[q];
            }
            for (int q = 0; q < 8; q++) kern[(3 * i + m) * 8 + q] = p[q];
        }
    }
}
extern "C" void coeffs(const double *v, int exact, double *o) {
    const KappaTables T{kern.data(), node.data()};
    if (exact)
        kappa_coeffs_quad<true>(T, v[0], v[1], v[2], v[3], v[4], v[5], o);
    else
        kappa_coeffs_quad<false>(T, v[0], v[1], v[2], v[3], v[4], v[5], o);
}
// F, G, H
static void synch(L x, L k[3]) {
    const L h = 0.09375L * std::min<L>(1, 1 / sqrtl(x));
    L a = 0.5L, b = 0.5L, c = 0.5L, d = 0.5L;
    for (int i = 1; i < 20000; i++) {
        const L t = i * h, u = expl(t / 3), w = 1 / u, ch = 0.5L * (u * u * u + w * w * w), sh = sinhl(t / 2);
        if (2 * x * sh * sh > 80 + 2 * t) break;
        const L e = expl(-2 * x * sh * sh), c13 = 0.5L * (u + w);
        a += e * 0.5L * (u * u * u * u * u + w * w * w * w * w) / ch;
        b += e * 0.5L * (u * u + w * w);
        c += e * c13;
        d += e * c13 / ch;
    }
    const L q = expl(-x);
    k[0] = q * x * h * a, k[1] = q * x * h * b, k[2] = q * (x * h * c + h * d);
}
extern "C" void reference(const double *v, double *o) {
    const L ne = v[0], Te = v[1], B = v[2], nu = v[3], kap = v[5];
    const bool th = kap <= 0;
    const L kw = (kap - 3) * Te, s0 = th ? 1 / Te : (kap + 1) / kw;
    const L lo = std::min<L>(0.5L * logl(1e-50L / s0), logl(1e-30L));
    const L hi = th ? 0.5L * logl(800 * Te * (800 * Te + 2)) : logl((1 + kw) * 10) + std::min<L>(45 / (kap - 2.34L), 600);
    const L n = ceill((hi - lo) / 0.02L), h = (hi - lo) / n, me = kMe, qe = kQe, c0 = kC;
    const L S = sinl(v[4]), as = fabsl(S), nuB = qe * B / (2 * PI * me * c0), X = nu / (1.5L * nuB * as);
    L na = 0, rv = 0, rq = 0, e[6] = {0};
    for (long i = 0; i <= (long)n; i++) {
        const L p = expl(lo + i * h), g = sqrtl(1 + p * p), gm1 = p * p / (g + 1), w = i == (long)n ? 0.5L : 1;
        const L q = w * (th ? expl(-gm1 / Te) : expl(-(kap + 1) * log1pl(gm1 / kw))), sl = th ? 1 / Te : (kap + 1) / (kw + gm1);
        const L N = p * p * p * q, D = (p / g - p * p * p * sl) * q, f = p * p * p * (2 * g - 1 / g) * q, c = kap - 3;
        na += N, rv += p * p * asinhl(p) / g * q, rq += f;
        if (i == (long)n && !th) rq += 2 * f * (c * h / 12 - c * c * c * h * h * h / 720);  // Euler-Maclaurin
        if (X / (g * g) < 3000) {
            L k[3];
            synch(X / (g * g), k);
            k[2] /= g;
            for (int j = 0; j < 3; j++) e[j] += N * k[j], e[3 + j] += D * k[j];
        }
    }
    const L x = Te * sqrtl(sqrtl(2) * as * 1000 * nuB / nu), t = powl(x / 120, 20);
    L f = 2.011L * expl(-powl(x, 1.035L) / 4.7L) - cosl(x / 2) * expl(-powl(x, 1.2L) / 2.73L) - 0.011L * expl(-x / 47.2L);
    if (x > 1) f += (0.011L * expl(-x / 47.2L) - powl(2, -1 / 3.L) * powl(3, -23 / 6.L) * 1e4L * PI * powl(x, -8 / 3.L)) * t / (1 + t);
    const L cc = cosl(v[4]), A = ne * sqrtl(3) * qe * qe * qe * B * as / (4 * PI * me * c0 * c0) / na, ab = -A / (2 * nu * nu * me);
    L r[8] = {A * e[0], A * e[1], A * 4 / 3 * (cc / S) * e[2], ab * e[3], ab * e[4], ab * 4 / 3 * (cc / S) * e[5],
              ne * qe * qe * nuB * nuB * S * S / (me * c0 * nu * nu * nu) * f * rq / na,
              2 * ne * qe * qe * nuB * cc / (me * c0 * nu * nu) * (1 - 0.11L * log1pl(0.035L * x)) * rv / na};
    for (int j = 0; j < 6; j += 3) {  // Q and V inside the light cone
        const L pq = r[j] > 0 ? sqrtl(r[j + 1] * r[j + 1] + r[j + 2] * r[j + 2]) / r[j] : 0;
        if (pq > 1) r[j + 1] /= pq, r[j + 2] /= pq;
    }
    for (int j = 0; j < 8; j++) o[j] = j < 6 && !(r[0] > 1e-250L) ? 0 : (double)r[j];
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = str(tmp_path_factory.mktemp("kappa"))
    with open(os.path.join(__graft_entry__.ROOT, "paper_2302_02733_gb300", "csrc", "kappa.cuh")) as f:
        text = f.read().replace('#include "rt_common.cuh"', "").replace("#pragma once", "")
    for name, body in (("kappa_host.h", text), ("k.cpp", SRC)):
        with open(os.path.join(d, name), "w") as f:
            f.write(body)
    r = subprocess.run([cxx, "-std=c++17", "-O2", "-shared", "-fPIC", "-o", os.path.join(d, "k.so"), os.path.join(d, "k.cpp")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(os.path.join(d, "k.so"))
    lib.tables()
    dp = ctypes.POINTER(ctypes.c_double)

    def call(row, exact=None):
        v, out = np.array(row, dtype=np.float64), np.zeros(8)
        args = (v.ctypes.data_as(dp),) + (() if exact is None else (int(exact),)) + (out.ctypes.data_as(dp),)
        (lib.reference if exact is None else lib.coeffs)(*args)
        return out

    return call


def field(X, th, nu=230e9):
    return nu / (1.5 * X * math.sin(th)) * 2 * math.pi * ME * C / E


def check(host, Te, X, th, kappa):
    row = (1e5, Te, field(X, th), 230e9, th, kappa)
    ref = host(row)
    tol = np.array([2e-9] * 3 + [2e-9 + 1e-14 / (Te * X)] * 3 + [1e-13] * 2)
    for exact in (False, True):
        got = host(row, exact)
        assert (np.abs(got - ref) <= tol * np.abs(ref)).all(), (row, exact, got, ref)


@pytest.mark.parametrize("kappa", [0.0, 3.1, 4.5, 12.0, 25.0, 50.0, 98.0])
def test_cold_electrons(host, kappa):
    """Electrons whose momenta lie at and below the first tabulated node, p = 1e-4: nothing of the
    distribution is lost there."""
    for Te in (1.9e-5, 1e-6, 1e-8, 1e-10, 6e-12, 1e-13):
        check(host, Te, 10.0, 1.0, kappa)
    for Te in (1e-30, 1e-100, 1e-300, 5e-324):  # finite, and the rotativities those of electrons at rest
        out = host((1e5, Te, field(10.0, 1.0), 230e9, 1.0, kappa), False)
        assert np.isfinite(out).all()
        rest = host((1e5, 1e-13, field(10.0, 1.0), 230e9, 1.0, 0.0))
        assert abs(out[7] - rest[7]) <= 1e-6 * abs(rest[7])


def test_unbounded_distributions_give_zeros(host):
    """Infinite or overflowing widths: zeros, as for other rows outside, and no endless sum."""
    for Te, kappa in ((math.inf, 0.0), (math.inf, 4.5), (1e160, 0.0), (1e200, 4.5), (1.0, math.inf), (1e200, 1e200)):
        assert (host((1e5, Te, 10.0, 230e9, 1.0, kappa), False) == 0.0).all(), (Te, kappa)


@pytest.mark.parametrize("kappa", [3.1, 4.5, 8.0, 12.0])
def test_power_law_tail_of_cold_electrons(host, kappa):
    """Emission of the tail far above a cold distribution's own peak: the sum does not end at the first of
    the two."""
    for Te in (1.9e-5, 1e-6, 1e-7, 1e-8, 1e-9):
        for X in (100.0, 600.0, 2000.0):
            check(host, Te, X, 1.0, kappa)


@pytest.mark.parametrize("kappa", [99.0, 1e3, 1e4, 1e6, 1e9])
def test_large_kappa(host, kappa):
    """Toward the Maxwell-Juttner limit the distribution's logarithm is kappa times a small number: no digits
    are lost to the power. At Theta_e of 20 and above what lies below the first node is under 1e-14."""
    for Te in (20.0, 300.0):
        check(host, Te, 10.0, 1.0, kappa)
