"""The FP64 tables of the thermal rotativities (csrc/thermtab.cuh), compiled for the CPU, filled from long
double values at their nodes and checked between them over every segment, at its ends too: K0/K2, K1/K2 and
g(X) to 2e-15 of their value, f(X) to 2e-15 of its terms (2.5 roundings of a node's value, some 10 of
the coefficients, 2 of the evaluation; 1e-16 each). Then what lies outside the tables. No GPU is used."""
import os
import shutil
import subprocess
import tempfile

import pytest

import __graft_entry__  # noqa: F401  (puts the repo root on sys.path)

SRC = r"""
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>
#define __device__
#define __forceinline__ inline
typedef long double L;
static const L PI = 3.14159265358979323846264338327950288L;
static double cospi(double x) { return (double)cosl(PI * x); }
static long long __double_as_longlong(double d) { long long x; std::memcpy(&x, &d, 8); return x; }
static double __longlong_as_double(long long x) { double d; std::memcpy(&d, &x, 8); return d; }
#include "thermtab.cuh"
using namespace prt;
typedef ThermTab T;
static void bessel(L Te, L v[2], L sc[2]) {
    const L z = 1 / Te, h = 0.09375L * std::min<L>(1, 1 / sqrtl(z));
    L s0 = 0.5L, s1 = 0.5L, s2 = 0.5L;
    for (int k = 1; k < 100000; k++) {
        const L t = k * h, sh = sinhl(t / 2), e = 2 * z * sh * sh;
        if (e > 2 * t + 60) break;
        const L w = expl(-e), c = coshl(t);
        s0 += w, s1 += w * c, s2 += w * (2 * c * c - 1);
    }
    sc[0] = v[0] = s0 / s2, sc[1] = v[1] = s1 / s2;
}
static void shcherbakov(L X, L v[2], L sc[2]) {
    const L a = 2.011L * expl(-powl(X, 1.035L) / 4.7L), b = cosl(X / 2) * expl(-powl(X, 1.2L) / 2.73L), c = 0.011L * expl(-X / 47.2L);
    v[0] = a - b - c, sc[0] = a + fabsl(b) + c;
    if (X > 1) {
        const L t = powl(X / 120, 20), w = t / (1 + t), d = powl(2, -1 / 3.L) * powl(3, -23 / 6.L) * 1e4L * PI * powl(X, -8 / 3.L);
        v[0] += (c - d) * w, sc[0] += (c + d) * w;
    }
    v[1] = 1 - 0.11L * log1pl(0.035L * X), sc[1] = 1 + 0.11L * log1pl(0.035L * X);
}
template <int D>
static void fill(double *tab, int n, int bits, int e0, void (*fn)(L, L *, L *)) {
    for (int i = 0; i < n; i++) {
        double f[2][D + 1], ch[D + 1];
        for (int j = 0; j <= D; j++) {
            L v[2], s[2];
            fn(T::at(i, bits, e0, cospi((j + 0.5) / (D + 1))), v, s);
            f[0][j] = (double)v[0], f[1][j] = (double)v[1];
        }
        for (int m = 0; m < 2; m++) {
            for (int k = 0; k <= D; k++) ch[k] = therm_chebyshev<D>(f[m], k);
            therm_powers<D>(ch, tab + (2 * i + m) * (D + 1));
        }
    }
}
int main() {
    std::vector<double> tab(T::size);
    fill<T::db>(&tab[T::bes], T::nb, 4, T::eb, bessel);
    fill<T::ds>(&tab[T::shc], T::ns, 4, T::es, shcherbakov);
    fill<T::ds>(&tab[T::shc + T::ns * 2 * (T::ds + 1)], T::nf, 6, T::ef, shcherbakov);
    long bad = 0, n = 0;
    double worst[4] = {0};
    auto check = [&](bool bes, double x) {
        double a, b, u;
        L v[2], s[2];
        const int i = bes ? therm_segment(x, 4, T::eb, u) : T::shc_segment(x, u);
        if (i < 0 || i >= (bes ? T::nb : T::ns + T::nf) || !(u >= -0.5 && u < 0.5)) {
            if (bad++ < 10) std::printf("%d %.17g: segment %d, u %g\n", bes, x, i, u);
            return;
        }
        if (bes)
            therm_eval<T::db>(&tab[T::bes + i * 2 * (T::db + 1)], u, a, b), bessel(x, v, s);
        else
            therm_eval<T::ds>(&tab[T::shc + i * 2 * (T::ds + 1)], u, a, b), shcherbakov(x, v, s);
        const double e[2] = {(double)(fabsl(a - v[0]) / s[0]), (double)(fabsl(b - v[1]) / s[1])};
        for (int m = 0; m < 2; m++) {
            worst[2 * !bes + m] = std::max(worst[2 * !bes + m], e[m]);
            if (!(e[m] <= 2e-15) && bad++ < 10) std::printf("%d function %d at %.6g: %.2e\n", bes, m, x, e[m]);
        }
        n++;
    };
    for (int k = 0; k < 60 * 64; k++)  // four stretches to each sixteenth of an octave
        for (double t : {0.0, 0.37, 0.999999999999}) check(true, ldexp(1.0 + ((k & 63) + t) / 64, T::eb + (k >> 6)));
    for (int k = 0; k < 44 * 64; k++)
        for (double t : {0.0, 0.21, 0.5, 0.83, 0.999999999999}) check(false, ldexp(1.0 + ((k & 63) + t) / 64, T::es + (k >> 6)));
    double u;
    for (double x : {0.0, 1e-300, std::nextafter(ldexp(1.0, -30), 0.0), ldexp(1.0, 14), 1e300, (double)INFINITY, (double)NAN})
        if (T::shc_segment(x, u) >= 0 && bad++ < 10) std::printf("%g in the table\n", x);
    std::printf("points %ld, worst %.2e %.2e %.2e %.2e, failures %ld\n", n, worst[0], worst[1], worst[2], worst[3], bad);
    return bad != 0;
}
"""


def test_tables_against_their_functions():
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    csrc = os.path.join(__graft_entry__.ROOT, "paper_2302_02733_gb300", "csrc")
    with tempfile.TemporaryDirectory() as d:
        src, exe = os.path.join(d, "t.cpp"), os.path.join(d, "t")
        with open(src, "w") as f:
            f.write(SRC)
        r = subprocess.run([cxx, "-std=c++17", "-O2", "-I", csrc, "-o", exe, src], capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
        r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
        print(r.stdout)
        assert r.returncode == 0, r.stdout + r.stderr
