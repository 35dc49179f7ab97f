"""The fixed-point face states (csrc/fixed_face.cuh, the FP64 form's
characteristic reconstruction) compiled for the host and compared with the
MEG7 procedure written out in long double (64 mantissa bits or more): the
reconstruction is exact on integers up to the projection's truncations (about
ten units of at most 2^-56 of the stencil's largest value) and the rounding of
each result to FP64, hence the tolerance 2^-53 |value| + 2^-52 scale."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2305_00762_gb300", "csrc")

SRC = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include "fixed_math.cuh"
using namespace gbr;
typedef long double R;
static R mm(R a, R b) { return (a < 0) != (b < 0) ? 0 : (fabsl(a) < fabsl(b) ? a : b); }
static R meg(const R* w, const R* e, int order)
{
    const R d0 = w[0] - w[2], d1 = w[1] - w[2], d2 = w[3] - w[2], d3 = w[4] - w[2];
    const R pl = order == 4 ? w[2] + e[2] / 2 + (e[1] - e[3]) / 24 + (d1 + d2) / 6
                            : w[2] + (420 * e[2] + 60 * (e[1] - e[3]) + 178 * (d1 + d2) + 3 * (d0 + d3)) / 840;
    const R mp = w[2] + mm(d2, -7 * d1);
    if ((pl - w[2]) * (pl - mp) <= 1e-40L) return pl;
    const R cm = 2 * (w[2] - 2 * w[1] + w[0]) - (e[2] - e[0]) / 2, c0 = 2 * (w[3] - 2 * w[2] + w[1]) - (e[3] - e[1]) / 2;
    const R cp = 2 * (w[4] - 2 * w[3] + w[2]) - (e[4] - e[2]) / 2;
    const R md = (w[2] + w[3]) / 2 - mm(c0, cp) / 2, ul = w[2] - 7 * d1, lc = (3 * w[2] - w[1]) / 2 + mm(c0, cm) * 4 / 3;
    const R lo = fmaxl(fminl(fminl(w[2], w[3]), md), fminl(fminl(w[2], ul), lc));
    const R hi = fminl(fmaxl(fmaxl(w[2], w[3]), md), fmaxl(fmaxl(w[2], ul), lc));
    return pl < lo ? lo : (pl > hi ? hi : pl);
}
struct Planes {  // the kernel's split planes of one face
    const double* const* u;
    int su;
    void operator()(int m, fx::Stencil& x) const
    {
        for (int k = 0; k < 12; ++k) {
            unsigned short e;
            fx::split(u[m][(k - 5) * su], x.m[k], e);
            x.e[k] = e;
        }
    }
};
template <int ORDER>
static int run(int mode, int stride)
{
    std::mt19937_64 g(7 + mode);
    std::uniform_real_distribution<double> U(-1, 1);
    double worst = 0;
    for (int it = 0; it < 20000; ++it) {
        double v[4][12 * 3];
        const double sc = mode == 2 ? std::pow(10.0, 6 * U(g)) : 1;
        for (int m = 0; m < 4; ++m) {
            const bool pos = m == 0 || m == 3;
            const double base = pos ? 1.5 + U(g) : (mode == 3 ? 30 * U(g) : U(g)), amp = std::pow(10.0, -8 * std::fabs(U(g)));
            const double jump = mode == 0 ? 0 : (pos ? std::fabs(U(g)) * 100 : U(g));
            const int at = (int)(g() % 13);
            for (int k = 0; k < 12; ++k) {
                double x = base + amp * (std::sin(0.7 * k + base) + 0.1 * U(g)) + (k < at ? jump : 0);
                if (mode == 4) x = pos ? 1.25 : (k % 2 ? 0.0 : -0.0);
                v[m][k * stride] = sc * (pos ? std::fabs(x) + 1e-3 : x);
            }
        }
        const double* u[4] = {v[0] + 5 * stride, v[1] + 5 * stride, v[2] + 5 * stride, v[3] + 5 * stride};
        const double rb = 0.5 * (u[0][0] + u[0][stride]), pb = 0.5 * (u[3][0] + u[3][stride]);
        const double c = std::sqrt(1.4 * pb / rb), rc = rb * c, ic2 = 1 / (c * c);
        fx::FaceStates o;
        fx::face_states<ORDER>(Planes{u, stride}, fx::pos(0.5 / rc), fx::pos(2 * rc), fx::pos(ic2), o);
        if (!o.ok) return std::printf("refused\n"), 1;
        R wl[4], wr[4], big[3] = {0, 0, 0};
        for (int f = 0; f < 4; ++f) {
            R q[12], e[12], a[5], b[5];
            for (int k = 0; k < 12; ++k) {
                const R r = v[0][k * stride], n = v[1][k * stride], t = v[2][k * stride], p = v[3][k * stride];
                q[k] = f == 0 ? p - (R)rc * n : f == 3 ? p + (R)rc * n : f == 1 ? r - (R)ic2 * p : t;
                const R s = f == 1 ? r + (R)ic2 * p : f == 2 ? fabsl(t) : p + (R)rc * fabsl(n);
                R& B = big[f == 1 ? 1 : f == 2 ? 2 : 0];
                B = fmaxl(B, s);
            }
            for (int k = 3; k < 9; ++k) e[k] = (45 * (q[k + 1] - q[k - 1]) - 9 * (q[k + 2] - q[k - 2]) + (q[k + 3] - q[k - 3])) / 60;
            for (int k = 0; k < 5; ++k) a[k] = q[3 + k], b[k] = e[3 + k];
            wl[f] = meg(a, b, ORDER);
            for (int k = 0; k < 5; ++k) a[k] = q[8 - k], b[k] = -e[8 - k];
            wr[f] = meg(a, b, ORDER);
        }
        const R y = 0.5 / rc, pl = (wl[0] + wl[3]) / 2, pr = (wr[0] + wr[3]) / 2;
        const R ref[8] = {pl, pr, (wl[3] - wl[0]) * y, (wr[3] - wr[0]) * y, wl[1] + pl * ic2, wr[1] + pr * ic2, wl[2], wr[2]};
        const R scale[4] = {big[0], big[0] * y * 2, big[1] + big[0] * ic2, big[2]};
        const double got[8] = {o.p[0], o.p[1], o.un[0], o.un[1], o.r[0], o.r[1], o.ut[0], o.ut[1]};
        for (int k = 0; k < 8; ++k) {
            const R tol = ldexpl(fabsl(ref[k]), -53) + ldexpl(scale[k / 2], -52);
            const R d = fabsl(ref[k] - (R)got[k]);
            if (!(d <= tol)) return std::printf("order %d mode %d value %d: %g off, %g allowed\n", ORDER, mode, k, (double)d, (double)tol), 1;
            if (tol > 0 && (double)(d / tol) > worst) worst = (double)(d / tol);
        }
    }
    std::printf("order %d mode %d: at most %.2f of the tolerance\n", ORDER, mode, worst);
    return 0;
}
// MEG7-cons: each functional of A and t carries at most seven truncations
// (alignment and six products) of one unit, 2^-59 of a scale at most 2^5 times
// the largest term; the limiter's bounds amplify them to at most 25 units and
// a returned sum takes two fields, hence 2^-53 |value| + 2^-48 of the largest
// term (the fields of one product more than cover theirs).
static int cons(int mode, int stride)
{
    std::mt19937_64 g(29 + mode);
    std::uniform_real_distribution<double> U(-1, 1);
    for (int it = 0; it < 20000; ++it) {
        double v[4][12 * 3];
        const double sc = mode == 2 ? std::pow(10.0, 5 * U(g)) : 1, mach = mode == 3 ? 20 : 1;
        const double r0 = 1.5 + U(g), p0 = 1.5 + U(g), u0 = mach * U(g), t0 = mach * U(g), amp = std::pow(10.0, -8 * std::fabs(U(g)));
        const double jump = mode ? 5 * std::fabs(U(g)) : 0;
        const int at = (int)(g() % 13);
        for (int k = 0; k < 12; ++k) {
            const double J = k < at ? jump : 0, r = r0 + J + amp * std::sin(k + r0), p = p0 + 3 * J + 0.3 * amp * U(g);
            const double n = mode == 4 ? 0 : u0 + 0.2 * J + amp * U(g), t = mode == 4 ? 0 : t0 + amp * U(g);
            v[0][k * stride] = sc * r, v[1][k * stride] = sc * r * n, v[2][k * stride] = sc * r * t;
            v[3][k * stride] = sc * (p / 0.4 + 0.5 * r * (n * n + t * t));
        }
        const double* u[4] = {v[0] + 5 * stride, v[1] + 5 * stride, v[2] + 5 * stride, v[3] + 5 * stride};
        const double c2 = 1.4 * p0 / r0, c = std::sqrt(c2);
        fx::ConsCoefs C;
        C.b1 = 0.4 / c2, C.b1u = C.b1 * u0, C.b1v = C.b1 * t0, C.b2 = 0.5 * C.b1 * (u0 * u0 + t0 * t0);
        C.uc = u0 / c, C.ic = 1 / c, C.v = t0;
        const Planes load{u, stride};
        fx::ConsStates o;
        fx::cons_states<7>(load, [&](int m) { fx::Stencil x; load(m, x); return fx::stencil_exponent(x); }, C, o);
        if (!o.ok) return std::printf("refused\n"), 1;
        R wl[4], wr[4], big = 0, big2 = 0;  // 2 w1, 2 w4, w2, w3
        for (int f = 0; f < 4; ++f) {
            R q[12], e[12], a[5], b[5];
            for (int k = 0; k < 12; ++k) {
                const R x0 = v[0][k * stride], x1 = v[1][k * stride], x2 = v[2][k * stride], x3 = v[3][k * stride];
                const R A = C.b2 * x0 - C.b1u * x1 - C.b1v * x2 + C.b1 * x3, t = C.uc * x0 - C.ic * x1;
                q[k] = f == 0 ? A + t : f == 1 ? A - t : f == 2 ? x0 - A : x2 - C.v * x0;
                for (R y : {C.b2 * x0, C.b1u * x1, C.b1v * x2, C.b1 * x3, C.uc * x0, C.ic * x1, x0}) big = fmaxl(big, fabsl(y));
                big2 = fmaxl(big2, fmaxl(fabsl(x2), fabsl(C.v * x0)));
            }
            for (int k = 3; k < 9; ++k) e[k] = (45 * (q[k + 1] - q[k - 1]) - 9 * (q[k + 2] - q[k - 2]) + (q[k + 3] - q[k - 3])) / 60;
            for (int k = 0; k < 5; ++k) a[k] = q[3 + k], b[k] = e[3 + k];
            wl[f] = meg(a, b, 7);
            for (int k = 0; k < 5; ++k) a[k] = q[8 - k], b[k] = -e[8 - k];
            wr[f] = meg(a, b, 7);
        }
        const R ref[8] = {(wl[0] + wl[1]) / 2 + wl[2], (wr[0] + wr[1]) / 2 + wr[2], (wl[0] + wl[1]) / 2, (wr[0] + wr[1]) / 2,
                          (wl[1] - wl[0]) / 2, (wr[1] - wr[0]) / 2, wl[3], wr[3]};
        const double got[8] = {o.r[0], o.r[1], o.s[0], o.s[1], o.d[0], o.d[1], o.w3[0], o.w3[1]};
        for (int k = 0; k < 8; ++k) {
            const R tol = ldexpl(fabsl(ref[k]), -53) + ldexpl(k < 6 ? big : big2, -48), d = fabsl(ref[k] - (R)got[k]);
            if (!(d <= tol)) return std::printf("cons mode %d value %d: %g off, %g allowed\n", mode, k, (double)d, (double)tol), 1;
        }
    }
    return 0;
}
static int limits()
{
    // integers round to double and back; infinities, NaN and overflowing scales are refused
    std::mt19937_64 g(1);
    for (int i = 0; i < 1000000; ++i) {
        const long long x = (long long)(g() >> (2 + g() % 62)) * (g() & 1 ? 1 : -1);
        const double d = fx::to_double(x, fx::kOne);
        if (std::fabs((double)((R)d - (R)x)) > std::ldexp(std::fabs((double)x), -53)) return std::printf("%lld -> %.17g\n", x, d), 1;
        long long m;
        unsigned short e;
        fx::split(d, m, e);
        if (fx::unsplit(m, e) != d) return std::printf("split %.17g\n", d), 1;
        if (std::fabs((double)x) < 9e15 && fx::aligned(m, e, fx::kOne) != x) return std::printf("back %lld\n", x), 1;
    }
    for (double d : {0.0, 1.0, -1.0, 1e-260, -1e260}) {
        long long m;
        unsigned short e;
        fx::split(d, m, e);
        if (fx::unsplit(m, e) != d) return std::printf("split %.17g\n", d), 1;
    }
    for (double d : {(double)INFINITY, 1e300, (double)NAN}) {
        long long m;
        unsigned short e;
        fx::split(d, m, e);
        if (!std::isnan(fx::unsplit(m, e))) return std::printf("split %.17g\n", d), 1;
    }
    if (fx::to_double(0, 700) != 0.0) return 1;
    for (double bad : {(double)INFINITY, (double)NAN, 1e300, -(double)INFINITY}) {
        double v[12];
        for (int m = 0; m < 4; ++m) {
            double w[4][12];
            for (int i = 0; i < 4; ++i)
                for (int k = 0; k < 12; ++k) w[i][k] = 1.0;
            w[m][3] = bad;
            const double* u[4] = {w[0] + 5, w[1] + 5, w[2] + 5, w[3] + 5};
            fx::FaceStates o;
            fx::face_states<7>(Planes{u, 1}, fx::pos(1 / 1.2), fx::pos(1.2), fx::pos(0.7), o);
            if (o.ok) return std::printf("%g accepted in plane %d\n", bad, m), 1;
        }
        (void)v;
    }
    return 0;
}
// The flux mean and the gradient against long double: exact but for the
// alignment (one unit of 2^-58 of the largest value each, times the weights'
// absolute sum over the divisor, at most 1.7 and 110) and the final rounding.
template <int ORDER>
static int sums(int mode)
{
    std::mt19937_64 g(11 + mode);
    std::uniform_real_distribution<double> U(-1, 1);
    const int w7[5] = {1052, -250, 38, 1, -1}, w4[5] = {1821, -461, 85, -4, -1};
    for (int it = 0; it < 50000; ++it) {
        double f[10];
        long long m[10];
        int ex[10];
        R big = 0, mean = 0, big7 = 0;
        for (int k = 0; k < 10; ++k) {
            f[k] = mode == 2 && k % 3 == 0 ? 0.0 : U(g) * std::pow(10.0, mode ? 8 * U(g) : 0.0);
            unsigned short e;
            fx::split(f[k], m[k], e);
            ex[k] = e;
            big = fmaxl(big, fabsl((R)f[k]));
            if (k < 7 && k != 3) big7 = fmaxl(big7, fabsl((R)f[k]));
        }
        for (int k = 0; k < 5; ++k) mean += (R)(ORDER == 4 ? w4 : w7)[k] * ((R)f[4 - k] + (R)f[5 + k]);
        mean /= ORDER == 4 ? 2880 : 1680;
        const double got = fx::recon_mean<ORDER>(m, ex);
        if (!(fabsl(got - mean) <= ldexpl(fabsl(mean), -53) + 4 * ldexpl(big, -57))) return std::printf("mean: %g %g\n", got, (double)mean), 1;
        long long m7[7];
        int e7[7];
        for (int k = 0; k < 7; ++k) m7[k] = m[k], e7[k] = ex[k];
        const R grad = 45 * ((R)f[4] - f[2]) - 9 * ((R)f[5] - f[1]) + ((R)f[6] - f[0]);
        const double gg = fx::grad60(m7, e7);
        if (!(fabsl(gg - grad) <= ldexpl(fabsl(grad), -53) + 400 * ldexpl(big7, -57))) return std::printf("gradient: %g %g\n", gg, (double)grad), 1;
    }
    return 0;
}
int main()
{
    int bad = limits();
    for (int mode = 0; mode < 5; ++mode) bad |= cons(mode, 1 + mode % 3);
    for (int mode = 0; mode < 3; ++mode) bad |= sums<7>(mode) | sums<4>(mode);
    for (int mode = 0; mode < 5; ++mode) bad |= run<7>(mode, 1 + mode % 3) | run<4>(mode, 1 + mode % 3);
    return bad;
}
"""


def test_fixed_point_face_states(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run([cxx, "-O2", "-std=c++17", "-Wno-unknown-pragmas", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
