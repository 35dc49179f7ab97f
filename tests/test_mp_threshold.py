"""The MP test's threshold (Eq. mp5Condition: a value is limited where (Phi^L -
Phi_j)(Phi^L - Phi^MP) > 1e-40) in the fixed-point face states, where densities,
pressures or the shear velocity are small enough for it to tell: states of scales
1 to 2^-90 against the procedure in long double, values whose product lies
within a factor of two of the threshold left out. Tolerances as in
tests/test_wide_face.py, 32 (MEG7-cons 128) units of 2^-53, here of the largest
terms of the stencil (a value may pass through zero). Where 1e-20 is less than
2^-54 of the speed of sound, a shear velocity may be off by the test's whole
effect, 1e-20 on each of two bounds."""
import os
import shutil
import subprocess

import pytest

from .test_wide_face import CSRC, SRC

# the procedure with the test, and whether a value is too close to the threshold
MEG = r"""
static bool g_tie;
static R meg(const R* w, const R* e, int order, R s)
{
    const R d0 = w[0] - w[2], d1 = w[1] - w[2], d2 = w[3] - w[2], d3 = w[4] - w[2];
    const R delta = order == 4 ? e[2] / 2 + (e[1] - e[3]) / 24 + (d1 + d2) / 6
                               : (420 * e[2] + 60 * (e[1] - e[3]) + 178 * (d1 + d2) + 3 * (d0 + d3)) / 840;
    const R pl = w[2] + delta, t = delta * (delta - mm(d2, -7 * d1)), thr = 1e-40L * s * s;
    if (t > thr / 2 && t < 2 * thr) g_tie = true;
    if (t <= thr) return pl;
"""
FILL = r"""
static void fill(Data& D, std::mt19937_64& g, int it, double scale)
{
    std::uniform_real_distribution<double> U(-1, 1);
    const int at = g() % 13, kind = it % 3;  // density and pressure small; the shear velocity; all three
    const double f = kind == 1 ? 1 : scale, fs = kind == 0 ? 1 : scale;
    const double jump = it % 4 ? std::pow(10.0, -12 * std::fabs(U(g))) : 0, wave = 0.3 * std::pow(10.0, -14 * std::fabs(U(g)));
    const double n0 = U(g), t0 = U(g);
    for (int k = 0; k < 12; ++k) {
        const double J = k < at ? jump : 0;
        D.v[0][k] = f * (1.1 + J + wave * U(g));
        D.v[3][k] = f * (0.9 + 1.4 * J + wave * U(g));
        D.v[1][k] = n0 + J + wave * U(g);
        D.v[2][k] = fs * (t0 + J + wave * U(g));
    }
    D.step = 1 + it % 3;
    D.normal = 1 + it % 2;
}
"""


def source():
    s = SRC
    a, b = s.index("static R meg("), s.index("    const R cm =")
    s = s[:a] + MEG + s[b:]
    a, b = s.index("static void fill("), s.index("template <int ORDER>\nstatic int prim")
    s = s[:a] + FILL + s[b:]
    s = s.replace("static void sides(const R* q, int order, R& l, R& r)", "static void sides(const R* q, int order, R s, R& l, R& r)")
    s = s.replace("meg(a, b, order)", "meg(a, b, order, s)")
    s = s.replace("        R w[4][2];\n", "        R w[4][2];\n        g_tie = false;\n")
    s = s.replace("sides(q, ORDER, w[f][0], w[f][1]);\n        }", "sides(q, ORDER, f < 2 ? 2 * (R)c * c : 1, w[f][0], w[f][1]);\n        }\n        if (g_tie) continue;")
    s = s.replace("sides(q, 7, w[f][0], w[f][1]);\n        }", "sides(q, 7, f < 2 ? 2 : 1, w[f][0], w[f][1]);\n        }\n        if (g_tie) continue;")
    # the terms of the whole stencil in the place of one cell's
    s = s.replace("        for (int s = 0; s < 2; ++s) {\n            const R p", "        double big[4] = {};\n"
                  "        for (int m = 0; m < 4; ++m)\n            for (int k = 0; k < 12; ++k) big[m] = std::max(big[m], std::fabs(D.v[m][k]));\n"
                  "        for (int s = 0; s < 2; ++s) {\n            const R p")
    s = s.replace("        for (int s = 0; s < 2; ++s) {\n            const double x0", "        double big[4] = {};\n"
                  "        for (int m = 0; m < 4; ++m)\n            for (int k = 0; k < 12; ++k) big[m] = std::max(big[m], std::fabs(D.v[m][k]));\n"
                  "        for (int s = 0; s < 2; ++s) {\n            const double x0")
    s = s.replace("off <= 32 * std::ldexp(scale[m], -53)", "off <= 32 * std::ldexp(scale[m], -53) + (m == 2 && 1e-20 < c * 0x1p-54 ? 2e-20 : 0)")
    s = s.replace("off <= 128 * std::ldexp(scale[m], -53)", "off <= 128 * std::ldexp(scale[m], -53) + (m == 3 && 1e-20 < rb / ic * 0x1p-54 ? 2e-20 : 0)")
    for a, b in (("std::fabs(D.v[3][5 + s])", "big[3]"), ("std::fabs(D.v[1][5 + s])", "big[1]"), ("std::fabs(D.v[2][5 + s])", "big[2]"),
                 ("D.v[0][5 + s]", "big[0]"), ("D.v[3][5 + s]", "big[3]")):
        assert a in s, a
        s = s.replace(a, b)
    s = s.replace("std::ldexp(1 + U(g), lr)", "std::ldexp(1 + U(g), -lr)").replace("lr <= 60; lr += lr < 12 ? 1 : 6", "lr <= 90; lr += 3")
    assert s.count("0x1p-54") == 2 and s.count("g_tie") == 6 and s.count("-lr") == 2 and s.count("order, s)") == 2
    return s


def test_states_of_small_scale(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(source())
    subprocess.run([cxx, "-O2", "-std=c++17", "-Wno-unknown-pragmas", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
