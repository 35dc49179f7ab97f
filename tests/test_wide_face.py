"""Face states beside jumps of many binary orders (csrc/fixed_face.cuh,
csrc/wide_face.cuh) compiled for the host, against the MEG7 procedure in long
double. The MP limiter bounds a face value by the cells beside the face, so its
error is measured against the terms of the cell on its side, not against the
largest value of the stencil: jumps by 1 to 2^60 (pressure; density as its
root), at every place of the stencil, rising and falling, at rest and moving,
with and without waves beside them.

Tolerances, in units of 2^-53 of those terms. MEG7-prim: a bound of the limiter
is 8 Phi_j - 7 Phi_{j-1} of values rounded by one unit each, and a state is the
mean of two fields or the sum of two: 32. MEG7-cons: a field is a sum of six
rounded products: 128."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2305_00762_gb300", "csrc")

SRC = r"""
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>
#include "wide_face.cuh"
using namespace gbr;
typedef long double R;
static R mm(R a, R b) { return (a < 0) != (b < 0) ? 0 : (fabsl(a) < fabsl(b) ? a : b); }
static R meg(const R* w, const R* e, int order)
{
    const R d0 = w[0] - w[2], d1 = w[1] - w[2], d2 = w[3] - w[2], d3 = w[4] - w[2];
    const R pl = order == 4 ? w[2] + e[2] / 2 + (e[1] - e[3]) / 24 + (d1 + d2) / 6
                            : w[2] + (420 * e[2] + 60 * (e[1] - e[3]) + 178 * (d1 + d2) + 3 * (d0 + d3)) / 840;
    const R cm = 2 * (w[2] - 2 * w[1] + w[0]) - (e[2] - e[0]) / 2, c0 = 2 * (w[3] - 2 * w[2] + w[1]) - (e[3] - e[1]) / 2;
    const R cp = 2 * (w[4] - 2 * w[3] + w[2]) - (e[4] - e[2]) / 2;
    const R md = (w[2] + w[3]) / 2 - mm(c0, cp) / 2, ul = w[2] - 7 * d1, lc = (3 * w[2] - w[1]) / 2 + mm(c0, cm) * 4 / 3;
    const R lo = fmaxl(fminl(fminl(w[2], w[3]), md), fminl(fminl(w[2], ul), lc));
    const R hi = fminl(fmaxl(fmaxl(w[2], w[3]), md), fmaxl(fmaxl(w[2], ul), lc));
    return pl < lo ? lo : (pl > hi ? hi : pl);
}
static void sides(const R* q, int order, R& l, R& r)
{
    R e[12], a[5], b[5];
    for (int k = 3; k < 9; ++k) e[k] = (45 * (q[k + 1] - q[k - 1]) - 9 * (q[k + 2] - q[k - 2]) + (q[k + 3] - q[k - 3])) / 60;
    for (int k = 0; k < 5; ++k) a[k] = q[3 + k], b[k] = e[3 + k];
    l = meg(a, b, order);
    for (int k = 0; k < 5; ++k) a[k] = q[8 - k], b[k] = -e[8 - k];
    r = meg(a, b, order);
}
typedef fx::WideLanes::V Lanes;
static const fx::WideLanes four{};
// four variables of 12 cells as planes with a step, y-face order where `normal` is 2
struct Data {
    double v[4][12];
    long long m[4 * 36];
    unsigned short e[4 * 36];
    int step, normal;
    int at(int p) const { return (p == 1 ? normal : p == 2 ? 3 - normal : p) * 36; }
    void take()
    {
        for (int p = 0; p < 4; ++p)
            for (int k = 0; k < 12; ++k) fx::split(v[p][k], m[at(p) + k * step], e[at(p) + k * step]);
    }
    void operator()(int p, fx::Stencil& x) const
    {
        for (int k = 0; k < 12; ++k) x.m[k] = m[at(p) + k * step], x.e[k] = e[at(p) + k * step];
    }
    fx::Face face() const { return fx::Face{m + 5 * step, e + 5 * step, step, 36, normal}; }
};
static void fill(Data& D, std::mt19937_64& g, int it, double ratio)
{
    std::uniform_real_distribution<double> U(-1, 1);
    const int at = 1 + g() % 11;
    const bool falling = g() & 1;
    const double un = it % 3 ? U(g) : 0, ut = it % 4 ? 0.3 : 0, wave = it % 2 ? 0.03 * std::pow(10.0, -4 * std::fabs(U(g))) : 0;
    const double s = std::sqrt(ratio), c = std::sqrt(s);  // density, velocities
    for (int k = 0; k < 12; ++k) {
        const bool hi = (k < at) == falling;
        const double w = wave * U(g);
        D.v[0][k] = (hi ? s : 1) * (1 + w) * 1.1;
        D.v[3][k] = (hi ? ratio : 1) * (1 + 1.4 * w) * 0.9;
        D.v[1][k] = un * (hi ? c : 1) * (1 + 0.5 * w);
        D.v[2][k] = ut * (hi ? c : 1) * (1 + w);
    }
    D.step = 1 + it % 3;
    D.normal = 1 + it % 2;
}
template <int ORDER>
static int prim(int lr)
{
    std::mt19937_64 g(5 + lr);
    std::uniform_real_distribution<double> U(0, 1);
    double worst = 0;
    for (int it = 0; it < 6000; ++it) {
        Data D;
        fill(D, g, it, std::ldexp(1 + U(g), lr));
        D.take();
        const double gp = 1.4 * 0.5 * (D.v[3][5] + D.v[3][6]), rb = 0.5 * (D.v[0][5] + D.v[0][6]);
        const double y = fx::rsqrt(gp * rb), c = gp * y, rc = rb * c, ic = rb * y, ic2 = ic * ic;
        fx::FaceStates o;
        fx::face_states<ORDER>(D, fx::pos(0.5 * y), fx::pos(2 * rc), fx::pos(ic2), o);
        if (!o.ok) return std::printf("refused\n"), 1;
        if (o.wide) {
            Lanes r, u, p;
            fx::wide_states<ORDER>(four, D.face(), 1.4, r, u, p);
            for (int s = 0; s < 2; ++s) o.r[s] = r.x[s], o.un[s] = u.x[s], o.p[s] = p.x[s];
        }
        if (o.wide_ut) {
            const Lanes t = fx::wide_shear<ORDER>(four, D.face());
            for (int s = 0; s < 2; ++s) o.ut[s] = t.x[s];
        }
        R w[4][2];
        for (int f = 0; f < 4; ++f) {
            R q[12];
            for (int k = 0; k < 12; ++k) {
                const R r = D.v[0][k], n = D.v[1][k], t = D.v[2][k], p = D.v[3][k];
                q[k] = f == 0 ? p - (R)rc * n : f == 1 ? p + (R)rc * n : f == 2 ? r - (R)ic2 * p : t;
            }
            sides(q, ORDER, w[f][0], w[f][1]);
        }
        for (int s = 0; s < 2; ++s) {
            const R p = (w[0][s] + w[1][s]) / 2, un = (w[1][s] - w[0][s]) * (R)0.5 * y, r = w[2][s] + p * (R)ic2;
            const double terms = std::fabs(D.v[3][5 + s]) + rc * std::fabs(D.v[1][5 + s]);
            const R ref[4] = {r, un, w[3][s], p};
            const double got[4] = {o.r[s], o.un[s], o.ut[s], o.p[s]};
            const double scale[4] = {D.v[0][5 + s] + terms * ic2, terms * y, std::fabs(D.v[2][5 + s]), terms};
            for (int m = 0; m < 4; ++m) {
                const double off = std::fabs((double)((R)got[m] - ref[m]));
                if (!(off <= 32 * std::ldexp(scale[m], -53)))
                    return std::printf("order %d, jump 2^%d, value %d side %d: %.3g of its terms off\n", ORDER, lr, m, s, off / scale[m]), 1;
                if (scale[m] > 0) worst = std::max(worst, off / std::ldexp(scale[m], -53));
            }
        }
    }
    std::printf("order %d, jump 2^%d: %.1f units\n", ORDER, lr, worst);
    return 0;
}
static int cons(int lr)
{
    std::mt19937_64 g(77 + lr);
    std::uniform_real_distribution<double> U(0, 1);
    double worst = 0;
    for (int it = 0; it < 6000; ++it) {
        Data D;
        fill(D, g, it, std::ldexp(1 + U(g), lr));
        const double gp = 1.4 * 0.5 * (D.v[3][5] + D.v[3][6]), rb = 0.5 * (D.v[0][5] + D.v[0][6]);
        const double y = fx::rsqrt(gp * rb), ic = rb * y;
        fx::ConsCoefs C;
        C.v = 0.5 * (D.v[2][5] + D.v[2][6]);
        const double u = 0.5 * (D.v[1][5] + D.v[1][6]);
        C.b1 = 0.4 * ic * ic, C.b1u = C.b1 * u, C.b1v = C.b1 * C.v, C.b2 = 0.5 * C.b1 * (u * u + C.v * C.v), C.uc = u * ic, C.ic = ic;
        for (int k = 0; k < 12; ++k) {
            const double r = D.v[0][k], n = D.v[1][k], t = D.v[2][k];
            D.v[3][k] = D.v[3][k] / 0.4 + 0.5 * r * (n * n + t * t), D.v[1][k] = r * n, D.v[2][k] = r * t;
        }
        D.take();
        fx::ConsStates o;
        fx::cons_states<7>(D, [&](int m) { fx::Stencil x; D(m, x); return fx::stencil_exponent(x); }, C, o);
        if (!o.ok) return std::printf("refused\n"), 1;
        if (o.wide_w3) {
            const Lanes t = fx::wide_cons_shear<7>(four, D.face(), C.v);
            for (int s = 0; s < 2; ++s) o.w3[s] = t.x[s];
        }
        if (o.wide) {
            Lanes r, t, d;
            fx::wide_cons_states<7>(four, D.face(), C, r, t, d);
            for (int s = 0; s < 2; ++s) o.r[s] = r.x[s], o.s[s] = t.x[s], o.d[s] = d.x[s];
        }
        R w[4][2];
        for (int f = 0; f < 4; ++f) {
            R q[12];
            for (int k = 0; k < 12; ++k) {
                const R x0 = D.v[0][k], x1 = D.v[1][k], x2 = D.v[2][k], x3 = D.v[3][k];
                const R A = C.b2 * x0 - C.b1u * x1 - C.b1v * x2 + C.b1 * x3, t = C.uc * x0 - C.ic * x1;
                q[k] = f == 0 ? A + t : f == 1 ? A - t : f == 2 ? x0 - A : x2 - C.v * x0;
            }
            sides(q, 7, w[f][0], w[f][1]);
        }
        for (int s = 0; s < 2; ++s) {
            const double x0 = D.v[0][5 + s], x1 = std::fabs(D.v[1][5 + s]), x2 = std::fabs(D.v[2][5 + s]), x3 = D.v[3][5 + s];
            const double A = std::max({C.b2 * x0, std::fabs(C.b1u) * x1, std::fabs(C.b1v) * x2, C.b1 * x3, std::fabs(C.uc) * x0, ic * x1});
            const R S = (w[0][s] + w[1][s]) / 2, ref[4] = {S + w[2][s], S, (w[1][s] - w[0][s]) / 2, w[3][s]};
            const double got[4] = {o.r[s], o.s[s], o.d[s], o.w3[s]}, scale[4] = {std::max(x0, A), A, A, std::max(x2, std::fabs(C.v) * x0)};
            for (int m = 0; m < 4; ++m) {
                const double off = std::fabs((double)((R)got[m] - ref[m]));
                if (!(off <= 128 * std::ldexp(scale[m], -53)))
                    return std::printf("cons, jump 2^%d, value %d side %d: %.3g of its terms off\n", lr, m, s, off / scale[m]), 1;
                if (scale[m] > 0) worst = std::max(worst, off / std::ldexp(scale[m], -53));
            }
        }
    }
    std::printf("cons, jump 2^%d: %.1f units\n", lr, worst);
    return 0;
}
int main()
{
    int bad = 0;
    for (int lr = 0; lr <= 60; lr += lr < 12 ? 1 : 6) bad |= prim<7>(lr) | prim<4>(lr) | cons(lr);
    return bad;
}
"""


def test_states_keep_the_accuracy_of_their_own_cell(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run([cxx, "-O2", "-std=c++17", "-Wno-unknown-pragmas", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
