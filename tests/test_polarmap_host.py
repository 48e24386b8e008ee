"""The inverse of the FMKS grid's polar map (csrc/polarmap.cuh), compiled for the CPU and checked
against the map in long double, for exponents from 0.7 to 60 (some singular on the equator, some for
which the table's guess is too far off for the fourth-order step), blend weights of 0 .. 1 and angles from
pole to pole, dense about the equator: mu(y) is the angle asked for, and d theta / d X2 and theta_j -
theta_g are those at y, within the rounding of the terms they are sums of. With eps = 2^-53, f1 the slope
and ya = |2 y / xt|^alpha (relative error (alpha |ln| + 3) eps, once for the table's guess and once here):
- mu: 8 pi eps for the sums, 2 f1 eps for y, 4 N |y| ya (alpha |ln| + 3) eps, 2e-16 f1 for what the step
  leaves out;
- slope: eps times 16 of its terms, 4 N ya (alpha |ln| + 3) eps, the slope's change over the error of y,
  and the Taylor remainder, below 1e-16 |alpha - 3| f1 / |y| + 1e-15 as the step's own is below 1e-16 f1.
No GPU is used."""
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
#include <cstdlib>
#include <vector>
#define __device__
#define __forceinline__ inline
using std::max;
using std::min;
static void sincospi(double x, double *s, double *c) {
    const long double p = 3.14159265358979323846264338327950288L * x;
    *s = (double)sinl(p), *c = (double)cosl(p);
}
namespace prt {
constexpr double kPi = 3.14159265358979323846;
constexpr int kX2TabW = 64, kX2TabT = 1024;
}
#include "polarmap.cuh"
using namespace prt;
typedef long double L;
struct G { double hslope, poly_xt, poly_alpha, poly_norm; const double *x2_table; };
static const L PI = 3.14159265358979323846264338327950288L;
static void map(const G &g, L w, L y, L &mu, L &f1, L &dd, L &f2, L &ya) {
    const L s = sinl(2 * PI * y), c = cosl(2 * PI * y), o = 1 - (L)g.hslope, N = g.poly_norm, al = g.poly_alpha;
    ya = powl(fabsl(2 * y / g.poly_xt), al);
    const L g0 = PI * y - o * s / 2, g1 = PI - PI * o * c;
    dd = 2 * N * y * (1 + ya / (al + 1)) - g0;
    mu = g0 + w * dd;
    f1 = g1 + w * (2 * N * (1 + ya) - g1);
    const L g2 = 2 * PI * PI * o * s;
    f2 = g2 + w * (y != 0 ? 2 * N * ya * al / y - g2 : 0);
}
int main(int, char **v) {
    G g;
    g.poly_xt = atof(v[1]), g.poly_alpha = atof(v[2]), g.hslope = atof(v[3]);
    g.poly_norm = 0.5 * kPi / (1.0 + 1.0 / ((g.poly_alpha + 1.0) * std::pow(g.poly_xt, g.poly_alpha)));
    std::vector<double> tab(kX2TabW * kX2TabT);
    L m, f1, dd, f2, ya;
    for (int i = 0; i < kX2TabW * kX2TabT; i++) {
        const double w = double(i / kX2TabT) / (kX2TabW - 1), t = kPi * double(i % kX2TabT) / (kX2TabT - 1) - kPi / 2;
        double lo = -0.5, hi = 0.5;
        for (int k = 0; k < 56; k++) {
            const double c = (lo + hi) / 2;
            map(g, w, c, m, f1, dd, f2, ya);
            (m < t ? lo : hi) = c;
        }
        tab[i] = 0.5 + (lo + hi) / 2;
    }
    g.x2_table = tab.data();
    long n = 0, bad = 0;
    const L eps = ldexpl(1, -53);
    for (int a = 0; a <= 40; a++)
        for (int k = -5001; k <= 5001; k++) {
            const double w = a < 40 ? a * a / 1600.0 : 1.0, u = k / 5001.0;
            const double mu = (abs(k) % 3 ? u : std::pow(std::fabs(u), 5) * (u < 0 ? -1 : 1)) * (0.5 * kPi - 1e-9);
            double d1, d0;
            const double y = fmks_y64(g, w, mu + 0.5 * kPi, mu, d1, d0);
            map(g, w, y, m, f1, dd, f2, ya);
            const L ly = (y != 0 && ya > 0 ? fabsl(logl(ya)) : 0) + 3, N = g.poly_norm, ay = std::max(std::fabs(y), 1e-300);
            const L e0 = eps * (8 * PI + 2 * f1 + 4 * N * ay * ya * ly) + 2e-16L * f1;
            const L e1 = eps * (16 * (2 * PI + 2 * N * (1 + ya)) + 4 * N * ya * ly) + fabsl(f2) * e0 / f1 +
                         1e-16L * fabsl((L)g.poly_alpha - 3) * f1 / ay + 1e-15L;
            const L e2 = e0 + eps * 16 * PI + fabsl(f1) * e0 / f1 + (2 * N * (1 + ya) + 2 * PI) * e0 / f1 + e1 * 3e-5L;
            n++;
            if (!(fabsl(m - mu) <= e0 && fabsl(d1 - f1) <= e1 && fabsl(d0 - dd) <= e2) && bad++ < 10)
                std::printf("w %.4f mu %.6e y %.6e: mu off %.2Le of %.2Le, slope %.2Le of %.2Le, dd %.2Le of %.2Le\n", w, mu, y,
                            fabsl(m - mu), e0, fabsl(d1 - f1), e1, fabsl(d0 - dd), e2);
        }
    std::printf("points %ld failures %ld\n", n, bad);
    return bad != 0;
}
"""


@pytest.mark.parametrize("xt,alpha,hslope", [(0.82, 14.0, 0.3), (0.9, 2.0, 1.0), (0.7, 4.0, 0.5), (0.82, 60.0, 0.1),
                                             (0.9, 1.0, 1.0), (0.9, 1.0, 0.3), (0.7, 3.0, 0.5), (0.6, 0.7, 0.6)])
def test_polar_map_inverse(xt, alpha, hslope):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    csrc = os.path.join(__graft_entry__.ROOT, "paper_2302_02733_gb300", "csrc")
    with tempfile.TemporaryDirectory() as d:
        src, exe = os.path.join(d, "map.cpp"), os.path.join(d, "map")
        with open(src, "w") as f:
            f.write(SRC)
        r = subprocess.run([cxx, "-std=c++17", "-O2", "-I", d, "-I", csrc, "-o", exe, src], capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
        r = subprocess.run([exe, str(xt), str(alpha), str(hslope)], capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stdout + r.stderr
