"""The integer-pipe reciprocal and reciprocal square root (csrc/fixed_math.cuh)
compiled for the host: within 0.51 ulp of the exact value, by the sign of an
exact residual (the correction keeps 62 bits, so a result differs from the
nearest double only within 2^-8 ulp of a tie), over the whole exponent range,
near powers of two and on the special values its comment names; and the
primitives and fluxes of a cell on integers against long double, products and
roots of mantissas among them. Tolerances: a velocity carries the reciprocal's
2^-61 and the truncation of a product kept to 58 bits at least (2^-57 |u|); the
pressure four truncations of one unit of 2^-58 of twice its largest term (2^-54 of
(gamma - 1) E); a flux the same of its own terms."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2305_00762_gb300", "csrc")

SRC = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "fixed_math.cuh"
using namespace gbr;
// |1 - x r| and |1 - x r^2| / 2 in units of r's last place (half a unit of relative 2^-53 .. 2^-52), from FMA residuals
static double off_rcp(double x, double r)
{
    const double e = std::fma(-x, r, 1.0);
    int k;
    const double f = std::frexp(r, &k);  // r = f 2^k, ulp 2^(k - 53): relative ulp 2^-53 / f
    return std::fabs(e) * std::fabs(f) * 9007199254740992.0;
}
static double off_rsqrt(double x, double r)
{
    const double s = r * r, se = std::fma(r, r, -s);  // r^2 = s + se exactly
    const double e = std::fma(-x, s, 1.0) - x * se;
    int k;
    const double f = std::frexp(r, &k);
    return 0.5 * std::fabs(e) * f * 9007199254740992.0;
}
// what the planes hold, exactly (59 bits); refused values as NaN
static long double value(const fx::Split& x)
{
    long long m;
    unsigned short e;
    fx::store(x, m, e);
    return e > fx::kExpMax ? NAN : ldexpl((long double)m, e - fx::kOne);
}
static int cells()
{
    std::mt19937_64 g(17);
    std::uniform_real_distribution<double> U(-1, 1);
    for (int i = 0; i < 300000; ++i) {
        const double sc = i % 3 == 0 ? std::pow(10.0, 60 * U(g)) : 1, vs = i % 4 == 0 ? std::pow(10.0, 20 * U(g)) : 1;
        const double r = sc * (1.0001 + U(g)), un = vs * U(g), ut = i % 5 == 0 ? 0 : vs * U(g), p = sc * vs * vs * std::pow(10.0, 3 * U(g));
        const double q[4] = {r, r * un, r * ut, p / 0.4 + 0.5 * r * (un * un + ut * ut)};
        fx::Cell c;
        fx::cell_of(q[0], q[1], q[2], q[3], fx::pos(0.4), c);
        const long double u = (long double)q[1] / q[0], v = (long double)q[2] / q[0], E = q[3];
        const long double P = (long double)0.4 * (E - (q[1] * u + q[2] * v) / 2), k = (q[1] * u + q[2] * v) / 2;
        const long double eu = ldexpl(fabsl(u), -53), ev = ldexpl(fabsl(v), -53), ep = ldexpl(0.4L * (E + k), -53) + ldexpl(fabsl(P), -53);
        const long double mom = fabsl((long double)q[1] * u) + fabsl((long double)q[1] * v) + fabsl((long double)q[2] * v);
        if (fabsl(value(c.u) - u) > eu || fabsl(value(c.v) - v) > ev || fabsl(value(c.p) - P) > ep || value(c.r) != q[0])
            return std::printf("primitives of %a %a %a %a\n", q[0], q[1], q[2], q[3]), 1;
        const long double f[4] = {value(fx::sum(c.ruu, c.p)), value(fx::product(c.ru, c.v)), value(fx::product(c.u, c.h)),
                             value(fx::sum(c.rvv, c.p))};
        const long double w[4] = {q[1] * u + P, q[1] * v, u * (E + P), q[2] * v + P};
        const long double tol[4] = {ep + ldexpl(mom, -52), ldexpl(mom, -52), (fabsl(u) * (E + fabsl(P))) * ldexpl(1, -51) + fabsl(u) * ep,
                                    ep + ldexpl(mom, -52)};
        for (int m = 0; m < 4; ++m)
            if (!(fabsl(f[m] - w[m]) <= tol[m])) return std::printf("flux %d of %a %a %a %a\n", m, q[0], q[1], q[2], q[3]), 1;
        // mantissa products and roots: truncated below 2^-62, rounded once
        const fx::Pos a = fx::pos(r), b = fx::pos(p);
        const double prod = fx::to_double(a * b), root = fx::to_double(fx::rsqrt(b)), inv = fx::to_double(fx::rcp(a));
        if (fabsl(prod - (long double)r * p) > ldexpl(0.51L * 2 * fabsl((long double)r * p), -53) || off_rsqrt(p, root) > 0.51 || off_rcp(r, inv) > 0.51)
            return std::printf("mantissas of %a %a\n", r, p), 1;
    }
    const double bad[6][4] = {{0, 1, 1, 1}, {-1, 1, 1, 1}, {NAN, 0, 0, 1}, {INFINITY, 0, 0, 1}, {1, NAN, 0, 1}, {1, 0, 0, INFINITY}};
    for (const auto& q : bad) {
        fx::Cell c;
        fx::cell_of(q[0], q[1], q[2], q[3], fx::pos(0.4), c);
        if (!std::isnan(value(c.p)) || !std::isnan(value(c.u))) return std::printf("accepted %g %g %g %g\n", q[0], q[1], q[2], q[3]), 1;
    }
    return 0;
}
int main()
{
    if (cells()) return 1;
    std::mt19937_64 g(3);
    double w1 = 0, w2 = 0;
    for (int i = 0; i < 6000000; ++i) {
        unsigned long long u = g();
        const unsigned long long e = i % 3 == 0 ? 60 + (u >> 52) % 1920 : 1021 + (u >> 52) % 5;
        u = (u & 0xFFFFFFFFFFFFFull) | (e << 52);
        if (i % 6 == 1) u &= ~0x3FFFFFFFFFFFFull;        // few bits set
        if (i % 6 == 2) u = (e << 52) - 1 - (u & 0xff);  // just below a power of two
        double x;
        memcpy(&x, &u, 8);
        const double a = off_rcp(x, fx::rcp(x)), b = off_rsqrt(x, fx::rsqrt(x)), c = off_rcp(-x, fx::rcp(-x));
        w1 = std::fmax(w1, std::fmax(a, c));
        w2 = std::fmax(w2, b);
    }
    std::printf("rcp %.4f ulp, rsqrt %.4f ulp\n", w1, w2);
    const double inf = INFINITY;
    const bool ok = fx::rcp(0.0) == inf && fx::rcp(-0.0) == -inf && fx::rcp(inf) == 0 && fx::rcp(1.0) == 1.0 &&
                    fx::rcp(-4.0) == -0.25 && std::isnan(fx::rcp(NAN)) && fx::rsqrt(0.0) == inf &&
                    fx::rsqrt(inf) == 0 && std::isnan(fx::rsqrt(-1.0)) && std::isnan(fx::rsqrt(NAN)) &&
                    std::isnan(fx::rsqrt(-inf)) && fx::rsqrt(4.0) == 0.5 && fx::rsqrt(5e-324) == inf;
    if (!ok) std::printf("special values\n");
    return !(ok && w1 <= 0.51 && w2 <= 0.51);
}
"""


def test_reciprocal_and_rsqrt(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run([cxx, "-O2", "-std=c++17", "-Wno-unknown-pragmas", "-I", CSRC, str(src), "-o", str(exe), "-lm"],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
