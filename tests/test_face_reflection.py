"""Reflecting a face's stencil (cells reversed, normal velocity negated) swaps its
states and negates their normal velocity, exactly in real arithmetic; in fixed
point (csrc/fixed_face.cuh) shifts and products round towards minus infinity or
with a centred offset, so bits differ. The difference, in units of 2^-53 of the
stencil's largest terms: a field's value carries up to four units of 2^-58 (three
of a product, one of the alignment), the limiter's bounds fifteen times that, a
state the mean of two fields and its own rounding, 2.4 units in all and 4.8 for
two; and no side is preferred: the mean of what is left of the sum of a velocity
and its mirror image stays below a tenth of a unit."""
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
#include "fixed_math.cuh"
using namespace gbr;
struct Load {
    const double (*v)[12];
    void operator()(int m, fx::Stencil& x) const
    {
        for (int k = 0; k < 12; ++k) {
            unsigned short e;
            fx::split(v[m][k], x.m[k], e);
            x.e[k] = e;
        }
    }
};
static fx::FaceStates states(const double (*v)[12])
{
    const double gp = 1.4 * 0.5 * (v[3][5] + v[3][6]), rb = 0.5 * (v[0][5] + v[0][6]), y = fx::rsqrt(gp * rb), c = gp * y, ic = rb * y;
    fx::FaceStates o;
    fx::face_states<7>(Load{v}, fx::pos(0.5 * y), fx::pos(2 * rb * c), fx::pos(ic * ic), o);
    return o;
}
int main()
{
    std::mt19937_64 g(11);
    std::uniform_real_distribution<double> U(-1, 1);
    double worst = 0, left = 0, n = 0;
    for (int it = 0; it < 40000; ++it) {
        double v[4][12], w[4][12];
        const int at = g() % 13;
        const double jump = it % 2 ? std::fabs(U(g)) : 0, wave = std::pow(10.0, -6 * std::fabs(U(g))), un = U(g), ut = U(g);
        for (int k = 0; k < 12; ++k) {
            const double J = k < at ? jump : 0;
            v[0][k] = 1.5 + J + 0.3 * wave * U(g);
            v[1][k] = un + J + wave * U(g);
            v[2][k] = ut + J + wave * U(g);
            v[3][k] = 1.2 + 2 * J + 0.3 * wave * U(g);
        }
        for (int m = 0; m < 4; ++m)
            for (int k = 0; k < 12; ++k) w[m][k] = m == 1 ? -v[m][11 - k] : v[m][11 - k];
        const fx::FaceStates a = states(v), b = states(w);
        if (!a.ok || !b.ok || a.wide != b.wide || a.wide_ut != b.wide_ut) return std::printf("flags differ\n"), 1;
        double big[4] = {};
        for (int m = 0; m < 4; ++m)
            for (int k = 0; k < 12; ++k) big[m] = std::max(big[m], std::fabs(v[m][k]));
        const double rc = std::sqrt(1.4 * big[3] * big[0]), p = big[3] + rc * big[1];
        const double scale[4] = {big[0] + p * big[0] / (1.4 * 0.8), p / std::sqrt(1.4 * 0.8 * 1.1), big[2], p};
        for (int s = 0; s < 2; ++s) {
            const double d[4] = {a.r[s] - b.r[1 - s], a.un[s] + b.un[1 - s], a.ut[s] - b.ut[1 - s], a.p[s] - b.p[1 - s]};
            for (int m = 0; m < 4; ++m) worst = std::max(worst, std::fabs(d[m]) / scale[m] * 0x1p53);
            left += d[1] / scale[1] * 0x1p53;
            n += 1;
        }
    }
    std::printf("%.2f units, %.4f left\n", worst, left / n);
    return !(worst <= 4.8 && std::fabs(left / n) <= 0.1);
}
"""


def test_reflected_states(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run([cxx, "-O2", "-std=c++17", "-Wno-unknown-pragmas", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
