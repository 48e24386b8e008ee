"""The fixed-point RK4 step of csrc/geofix.cuh, compiled for the CPU and checked against the same
step in long double (64 bits of significand or more) with the acceleration written independently,
from the metric's derivatives:
- along backward rays of several spins and inclinations, every step taken in fixed point is within
  half a unit in the last place of the FP64 result plus 2^-54 of the component's scale (the rounding
  of the final FP64 sum, and the increment's error), where the scale of a momentum component is the
  ray's largest momentum component in an orthonormal frame;
- few of those steps leave the form's bounds (those go to the FP64 form);
- on random states and step sizes, in and out of the bounds, null or not, no sum or shift of a step
  that reports success overflows;
- states outside the bounds (r < 1, on the axis, not finite) are refused.
No GPU is used."""
import os
import subprocess
import tempfile

import pytest

import __graft_entry__  # noqa: F401  (puts the repo root on sys.path)

SRC = r"""
#include <cstdint>
#include <cstring>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>
#include <algorithm>
#define __device__
#define __forceinline__ inline
#define __restrict__
static inline long long __double_as_longlong(double d) { long long x; std::memcpy(&x, &d, 8); return x; }
static inline double __longlong_as_double(long long x) { double d; std::memcpy(&d, &x, 8); return d; }
static inline unsigned __float_as_uint(float f) { unsigned u; std::memcpy(&u, &f, 4); return u; }
static inline float __uint_as_float(unsigned u) { float f; std::memcpy(&f, &u, 4); return f; }
static inline int __float_as_int(float f) { int i; std::memcpy(&i, &f, 4); return i; }
static inline float __int_as_float(int i) { float f; std::memcpy(&f, &i, 4); return f; }
static long misfits = 0;
#define FX_FITS(ok) do { if (!(ok)) misfits++; } while (0)
#include "geofix.cuh"
using namespace prt;
typedef long double L;
static const double PI = 3.14159265358979323846;
static std::vector<fx64> tab;

struct G { L g[4][4], gr[4][4], gt[4][4], inv[4][4]; };
static G metric(L a, L r, L th) {
    G m; std::memset(&m, 0, sizeof m);
    const L s = sinl(th), c = cosl(th), s2 = s * s, sg = r * r + a * a * c * c, q = 2 * r / sg;
    const L qr = 2 / sg - 4 * r * r / (sg * sg), qt = 4 * a * a * r * s * c / (sg * sg), st = -2 * a * a * s * c;
    auto put = [](L x[4][4], int i, int j, L v) { x[i][j] = x[j][i] = v; };
    put(m.g, 0, 0, q - 1); put(m.g, 0, 1, q); put(m.g, 0, 3, -a * s2 * q); put(m.g, 1, 1, 1 + q);
    put(m.g, 1, 3, -a * s2 * (1 + q)); put(m.g, 2, 2, sg); put(m.g, 3, 3, s2 * (sg + a * a * s2 * (1 + q)));
    put(m.gr, 0, 0, qr); put(m.gr, 0, 1, qr); put(m.gr, 0, 3, -a * s2 * qr); put(m.gr, 1, 1, qr);
    put(m.gr, 1, 3, -a * s2 * qr); put(m.gr, 2, 2, 2 * r); put(m.gr, 3, 3, s2 * (2 * r + a * a * s2 * qr));
    put(m.gt, 0, 0, qt); put(m.gt, 0, 1, qt); put(m.gt, 0, 3, -a * (2 * s * c * q + s2 * qt)); put(m.gt, 1, 1, qt);
    put(m.gt, 1, 3, -a * (2 * s * c * (1 + q) + s2 * qt)); put(m.gt, 2, 2, st);
    put(m.gt, 3, 3, 2 * s * c * (sg + a * a * s2 * (1 + q)) + s2 * (st + a * a * (2 * s * c * (1 + q) + s2 * qt)));
    put(m.inv, 0, 0, -(1 + q)); put(m.inv, 0, 1, q); put(m.inv, 1, 1, (r * r - 2 * r + a * a) / sg); put(m.inv, 1, 3, a / sg);
    put(m.inv, 2, 2, 1 / sg); put(m.inv, 3, 3, 1 / (sg * s2));
    return m;
}
// rates of (r, theta, phi, W = K^t + K^r, K^r, K^theta, K^phi)
static void rate(L a, const L y[7], L k[7]) {
    const G m = metric(a, y[0], y[1]);
    const L K[4] = {y[3] - y[4], y[4], y[5], y[6]};
    L F[4], acc[4];
    for (int n = 0; n < 4; n++) {
        F[n] = 0;
        for (int b = 0; b < 4; b++) F[n] += (K[1] * m.gr[n][b] + K[2] * m.gt[n][b]) * K[b];
    }
    for (int i = 0; i < 4; i++)
        for (int j = 0; j < 4; j++) {
            F[1] -= m.gr[i][j] * K[i] * K[j] / 2;
            F[2] -= m.gt[i][j] * K[i] * K[j] / 2;
        }
    for (int i = 0; i < 4; i++) {
        acc[i] = 0;
        for (int j = 0; j < 4; j++) acc[i] -= m.inv[i][j] * F[j];
    }
    k[0] = y[4]; k[1] = y[5]; k[2] = y[6]; k[3] = acc[0] + acc[1]; k[4] = acc[1]; k[5] = acc[2]; k[6] = acc[3];
}
static void rk4(L a, L h, const double y0[7], L out[7]) {
    L y[7], k[4][7], z[7];
    for (int i = 0; i < 7; i++) y[i] = y0[i];
    rate(a, y, k[0]);
    for (int s = 1; s < 4; s++) {
        for (int i = 0; i < 7; i++) z[i] = y[i] + (s == 3 ? h : h / 2) * k[s - 1][i];
        rate(a, z, k[s]);
    }
    for (int i = 0; i < 7; i++) out[i] = y[i] + h / 6 * (k[0][i] + 2 * k[1][i] + 2 * k[2][i] + k[3][i]);
}
static double step_size(double eps, const double y[7]) {
    const double tt = std::max(std::min(y[1], PI - y[1]), 1e-2);
    return eps / (std::fabs(y[4]) / y[0] + std::fabs(y[5]) / tt + std::fabs(y[6]));
}
static int rays(double a, double incl, int N) {
    const double rc = 1000.0, rh = 1 + std::sqrt(1 - a * a);
    long steps = 0, out = 0, bad = 0;
    for (int iy = 0; iy < N; iy++)
        for (int ix = 0; ix < N; ix++) {
            // a past-directed null vector toward (x, y) at the camera: K_th and K_ph from the image
            // position, K^r < 0 of unit size, K^t from the null condition
            const double x = ((ix + 0.5) / N - 0.5) * 40, yy = ((iy + 0.5) / N - 0.5) * 40, th = incl * PI / 180;
            const G m = metric(a, rc, th);
            L K[4] = {0, -1, -yy / (rc * rc), x / (rc * rc * std::sin(th))};
            L B = 0, C = 0;
            for (int i = 1; i < 4; i++) {
                B += m.g[0][i] * K[i];
                for (int j = 1; j < 4; j++) C += m.g[i][j] * K[i] * K[j];
            }
            K[0] = (-B + sqrtl(B * B - m.g[0][0] * C)) / m.g[0][0];
            double y[7] = {rc, th, 0, (double)(K[0] + K[1]), (double)K[1], (double)K[2], (double)K[3]};
            for (int n = 0; n < 20000; n++) {
                const double h = step_size(0.05, y);
                double o[7];
                L ref[7];
                rk4(a, h, y, ref);
                const long m0 = misfits;
                steps++;
                if (!fx_step(tab.data(), a, h, y, o)) {
                    out++;
                    misfits = m0;
                    for (int i = 0; i < 7; i++) o[i] = (double)ref[i];
                } else {
                    const double s = std::sin(y[1]);
                    const double kk = std::max(std::max(std::fabs(y[3]), std::fabs(y[4])),
                                               y[0] * std::max(std::fabs(y[5]), s * std::fabs(y[6])));
                    const double sc[7] = {y[0], 1, 1 / s, kk, kk, kk / y[0], kk / (y[0] * s)};
                    for (int i = 0; i < 7; i++) {
                        const double ulp = std::ldexp(1.0, std::ilogb((double)ref[i] == 0 ? 1e-300 : (double)ref[i]) - 52);
                        if (!(fabsl((L)o[i] - ref[i]) <= 0.5L * ulp + std::ldexp(sc[i], -54)) && bad++ < 10)
                            std::printf("component %d off by %.3Le (scale %.3e, ulp %.3e) r %.6f theta %.6f\n", i,
                                        (L)o[i] - ref[i], sc[i], ulp, y[0], y[1]);
                    }
                }
                std::memcpy(y, o, sizeof y);
                if (y[1] < 0) { y[1] = -y[1]; y[2] += PI; y[5] = -y[5]; }
                else if (y[1] > PI) { y[1] = 2 * PI - y[1]; y[2] += PI; y[5] = -y[5]; }
                if (y[0] < 1.05 * rh || (y[0] > rc && y[4] > 0)) break;
            }
        }
    std::printf("steps %ld outside %ld bad %ld misfits %ld\n", steps, out, bad, misfits);
    return bad || misfits || out > steps / 50;
}
static uint64_t sd = 88172645463325252ull;
static double U() { sd ^= sd << 13; sd ^= sd >> 7; sd ^= sd << 17; return (sd >> 11) * (1.0 / 9007199254740992.0); }
static int box(long n) {
    long done = 0;
    for (long k = 0; k < n; k++) {
        const double a = (2 * U() - 1) * (U() < 0.3 ? 0.99999 : 0.95), rh = 1 + std::sqrt(1 - a * a);
        double y[7], o[7];
        y[0] = U() < 0.5 ? rh * (0.98 + 2 * U()) : std::pow(10.0, 4 * U()) * rh;
        y[1] = U() < 0.3 ? std::pow(10.0, -4 * U()) : U() * PI;
        if (U() < 0.5) y[1] = PI - y[1];
        y[2] = 6 * U();
        const double sc = std::pow(10.0, 4 * U() - 2), s = std::sin(y[1]);
        y[3] = (2 * U() - 1) * sc * (U() < 0.3 ? 40 : 1);
        y[4] = (2 * U() - 1) * sc;
        y[5] = (2 * U() - 1) * sc / y[0];
        y[6] = (2 * U() - 1) * sc / y[0] / (U() < 0.7 ? s : std::sqrt(s));
        const double eps = U() < 0.7 ? 0.05 : std::pow(10.0, 3 * U() - 3);
        const long m0 = misfits;
        if (fx_step(tab.data(), a, step_size(eps, y), y, o))
            done++;
        else
            misfits = m0;
    }
    std::printf("steps %ld taken %ld misfits %ld\n", n, done, misfits);
    return misfits != 0 || done < n / 2;
}
static int refused() {
    const double nan = NAN, inf = INFINITY;
    const double good[7] = {10, 1, 0, -0.2, -0.9, 0.02, 0.03};
    double o[7];
    int bad = !fx_step(tab.data(), 0.9, 0.4, good, o);
    auto no = [&](int i, double v) {
        double y[7];
        std::memcpy(y, good, sizeof y);
        y[i] = v;
        if (fx_step(tab.data(), 0.9, 0.4, y, o)) std::printf("accepted %d %g\n", i, v), bad = 1;
    };
    for (double v : {nan, inf, -inf, 0.9, 0.0, -3.0, 1e300}) no(0, v);
    for (double v : {nan, inf, -inf, 0.0, 1e-4, PI, -0.5, 4.0, 7.5}) no(1, v);
    for (int i = 3; i < 7; i++)
        for (double v : {nan, inf, -inf, 1e300}) no(i, v);
    for (double h : {nan, inf, 1e300}) if (fx_step(tab.data(), 0.9, h, good, o)) std::printf("accepted h %g\n", h), bad = 1;
    return bad;
}
int main(int argc, char **argv) {
    for (int k = 0; k < kFxTab; k++)
        for (int j = 0; j < 2; j++)
            tab.push_back((fx64)llroundl((j ? cosl(k / 256.0L) : sinl(k / 256.0L)) * 4611686018427387904.0L));
    const char *what = argv[1];
    if (!std::strcmp(what, "box")) return box(atol(argv[2]));
    if (!std::strcmp(what, "refused")) return refused();
    return rays(atof(argv[2]), atof(argv[3]), atoi(argv[4]));
}
"""


@pytest.fixture(scope="module")
def exe():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    with tempfile.TemporaryDirectory() as d:
        src, out = os.path.join(d, "t.cpp"), os.path.join(d, "t")
        open(os.path.join(d, "cuda_runtime.h"), "w").close()
        open(src, "w").write(SRC)
        r = subprocess.run(["g++", "-O2", "-std=c++17", "-fwrapv", "-ffp-contract=off", "-I", d, "-I",
                            os.path.join(root, "paper_2302_02733_gb300", "csrc"), "-o", out, src],
                           capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
        yield out


@pytest.mark.parametrize("args", [("rays", "0.9375", "20", "6"), ("rays", "0", "60", "5"), ("rays", "-0.7", "110", "5"),
                                  ("rays", "0.998", "89", "5"), ("box", "400000"), ("refused",)])
def test_fixed_point_step(exe, args):
    r = subprocess.run([exe, *args], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
