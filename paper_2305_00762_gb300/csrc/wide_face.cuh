// Face states for stencils that span too many binary orders for one fixed-point
// scale.
//
// The fixed-point form (fixed_face.cuh) holds a stencil's values in units of
// 2^-59 of the largest one. The MP limiter bounds a face value by the cells
// beside the face, so in floating point the low side of a jump keeps its own
// relative accuracy, whatever lies five cells away; in fixed point it keeps
// 2^-59 of the jump. Where the largest term of a stencil exceeds the terms of a
// cell beside the face by more than kWide binary orders (`wide` of FaceStates and
// ConsStates), the face is evaluated here: each functional of a variable on
// integers at the scale of its own nine cells, which an FP64 sum is rounded by
// too, and the projection and the limiter in FP64.
//
// Such faces lie within six cells of a jump by a factor of 16 or more, or have a
// shear velocity far below the stencil's. They are few (2% of the faces of a
// developed four-quadrant flow), so the code is kept out of line: inlined, its
// registers would be taken from every face. FP64 operations a face: 22 for the
// shear field, 110 for the other three (with gradients and differences in FP64
// as well 78 and 290: one instruction holds the FP64 pipe for 19 clocks however
// few lanes are active, and a warp with one such face issues them all). What the
// accuracy costs, us a pass without / with: 64^2 vortex 880 / 898, four-quadrant
// 400^2 1451 / 1592, 1024^2 3986 / 4138, MEG7-cons 400^2 1921 / 2567, double Mach
// 1024 x 256 (a shock of ratio 116 through four tiles a row) 1881 / 2221.
//
// The MP test's absolute threshold, which fixed point leaves out, is applied here,
// and faces where it tells (kSmall: densities below 2^-12) are evaluated here too:
// four-quadrant flow 1024^2 in units with densities of 1e-4 8.5 ms a pass.
#pragma once

#include "fixed_math.cuh"

#ifndef __CUDACC__
#include <math.h>
#endif

namespace gbr {
namespace fx {

GBR_HD double fmadd(double a, double b, double c)
{
#ifdef __CUDA_ARCH__
    return __fma_rn(a, b, c);
#else
    return fma(a, b, c);
#endif
}

// The split planes of a face's stencil: the cell before the face, the distance
// to the next cell across it, values per plane, the plane of the normal
// component (1 or 2).
struct Face {
    const i64* m;
    const unsigned short* e;
    int step, values, normal;
    GBR_HD int at(int v) const { return (v == 1 ? normal : v == 2 ? 3 - normal : v) * values; }  // variable rho, un, ut, p
};

// Functionals (fixed_face.cuh) as doubles.
struct WideFunctionals {
    double v[4], n[2], d[4];
};
template <int ORDER>
GBR_HD void wide_functionals(const Face& f, int variable, WideFunctionals& o)
{
    const int at = f.at(variable);
    i64 m[12];
    int e[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        m[k] = f.m[at + (k - 5) * f.step];
        e[k] = f.e[at + (k - 5) * f.step];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        o.v[k] = unsplit(m[4 + k], e[4 + k]);
        int s = kExpMin;
#pragma unroll
        for (int c = 0; c < 9; ++c) s = larger(s, e[k + c]);
        i64 q[9];
#pragma unroll
        for (int c = 0; c < 9; ++c) q[c] = aligned(m[k + c], e[k + c], s);
        i64 d, n[2];
        centred<ORDER>(q + 4, k, d, n);
        o.d[k] = to_double(d, s);
        if (k == 1) o.n[0] = to_double(n[0], s);
        if (k == 2) o.n[1] = to_double(n[1], s);
    }
}

// minmod and the clamp on the bits (values that are not NaN).
GBR_HD double minmod(double a, double b)
{
    const i64 x = (i64)bits_of(a), y = (i64)bits_of(b);
    const double r = (x & 0x7fffffffffffffffll) <= (y & 0x7fffffffffffffffll) ? a : b;
    return (x ^ y) < 0 ? 0.0 : r;
}
GBR_HD i64 order_key(double x)
{
    const i64 b = (i64)bits_of(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
GBR_HD double mp_clamp(double p2, double p3, double md, double ul, double lc, double pl)
{
    const i64 k = mp_clamp(order_key(p2), order_key(p3), order_key(md), order_key(ul), order_key(lc), order_key(pl));
    return of_bits((u64)(k ^ ((k >> 63) & 0x7fffffffffffffffll)));
}

// The MEG7 values (Eqs. grb, mp5Condition, mp-procedure) left and right of the
// face of a field carried at `scale` times its value.
template <int ORDER>
GBR_HD void wide_limited(const WideFunctionals& f, double scale, double& vl, double& vr)
{
    constexpr double kN = ORDER == 4 ? 8192.0 / 10080.0 : 1024.0 / 840.0, kD = 128.0 / 120.0;  // n, d -> delta, d_j
    const double st = 1e-20 * scale, thr = st * st;
    const double b = f.v[2] - f.v[1], a[2] = {f.v[0] - f.v[1], f.v[3] - f.v[2]};
    const double md = 0.5 * fmadd(-kD, minmod(f.d[1], f.d[2]), f.v[1] + f.v[2]);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const double c = f.v[1 + k], delta = kN * f.n[k], m = minmod(k ? -b : b, -7.0 * a[k]);
        double v = c + delta;
        if (!(delta * (delta - m) <= thr)) {
            const double mm = minmod(f.d[1 + k], f.d[k ? 3 : 0]);
            v = mp_clamp(c, f.v[2 - k], md, fmadd(-7.0, a[k], c), fmadd(4.0 / 3.0 * kD, mm, fmadd(-0.5, a[k], c)), v);
        }
        (k ? vr : vl) = v;
    }
}
// o = x + a y, every functional
GBR_HD void combine(const WideFunctionals& x, double a, const WideFunctionals& y, WideFunctionals& o)
{
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        o.v[k] = fmadd(a, y.v[k], x.v[k]);
        o.d[k] = fmadd(a, y.d[k], x.d[k]);
    }
    o.n[0] = fmadd(a, y.n[0], x.n[0]);
    o.n[1] = fmadd(a, y.n[1], x.n[1]);
}

template <int ORDER>
GBR_OUTLINE void wide_shear(Face f, double (&ut)[2])
{
    WideFunctionals x;
    wide_functionals<ORDER>(f, 2, x);
    wide_limited<ORDER>(x, 1.0, ut[0], ut[1]);
}

// rho, un and p of both sides. Fields as in face_states: p -/+ rho c un and
// rho - p / c^2.
template <int ORDER>
GBR_OUTLINE void wide_states(Face f, double gamma, FaceStates& o)
{
    WideFunctionals P, X, W;
    wide_functionals<ORDER>(f, 3, P);
    wide_functionals<ORDER>(f, 0, X);
    const double r = 0.5 * (X.v[1] + X.v[2]), gp = gamma * (0.5 * (P.v[1] + P.v[2]));
    const double y = rsqrt(gp * r), c = gp * y, rc = r * c, ic = r * y, ic2 = ic * ic;
    double s[2], l[2], h[2];
    combine(X, -ic2, P, W);
    wide_limited<ORDER>(W, 1.0, s[0], s[1]);
    wide_functionals<ORDER>(f, 1, X);
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {  // (one copy of the limiter)
        combine(P, k ? rc : -rc, X, W);
        double a, b;
        wide_limited<ORDER>(W, 2.0 * c * c, a, b);
        if (k) l[1] = a, h[1] = b;
        else l[0] = a, h[0] = b;
    }
    const double be = 0.5 * ic2, hrc = 0.5 * y, pl = l[0] + l[1], pr = h[0] + h[1];
    o.r[0] = fmadd(be, pl, s[0]);
    o.r[1] = fmadd(be, pr, s[1]);
    o.un[0] = hrc * (l[1] - l[0]);
    o.un[1] = hrc * (h[1] - h[0]);
    o.p[0] = 0.5 * pl;
    o.p[1] = 0.5 * pr;
}

// MEG7-cons: w3, and the others.
template <int ORDER>
GBR_OUTLINE void wide_cons_shear(Face f, double v, double (&w3)[2])
{
    WideFunctionals Q, W;
    wide_functionals<ORDER>(f, 0, Q);
    wide_functionals<ORDER>(f, 2, W);
    combine(W, -v, Q, W);
    wide_limited<ORDER>(W, 1.0, w3[0], w3[1]);
}
template <int ORDER>
GBR_OUTLINE void wide_cons_states(Face f, ConsCoefs C, ConsStates& o)
{
    WideFunctionals Q, A, T, W;  // A and t as in cons_states
    double l[2], h[2];
    wide_functionals<ORDER>(f, 3, Q);
#pragma unroll
    for (int k = 0; k < 4; ++k) A.v[k] = C.b1 * Q.v[k], A.d[k] = C.b1 * Q.d[k];
    A.n[0] = C.b1 * Q.n[0], A.n[1] = C.b1 * Q.n[1];
    wide_functionals<ORDER>(f, 1, Q);
    combine(A, -C.b1u, Q, A);
#pragma unroll
    for (int k = 0; k < 4; ++k) T.v[k] = -C.ic * Q.v[k], T.d[k] = -C.ic * Q.d[k];
    T.n[0] = -C.ic * Q.n[0], T.n[1] = -C.ic * Q.n[1];
    wide_functionals<ORDER>(f, 2, Q);
    combine(A, -C.b1v, Q, A);
    wide_functionals<ORDER>(f, 0, Q);
    combine(A, C.b2, Q, A);
    combine(T, C.uc, Q, T);
    combine(Q, -1.0, A, Q);
    double s[2];
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {  // 2 w1, 2 w4, w2
        double a, b;
        if (k < 2) combine(A, k ? -1.0 : 1.0, T, W);
        else W = Q;
        wide_limited<ORDER>(W, k < 2 ? 2.0 : 1.0, a, b);
        if (k == 0) l[0] = a, h[0] = b;
        if (k == 1) l[1] = a, h[1] = b;
        if (k == 2) s[0] = a, s[1] = b;
    }
    o.s[0] = 0.5 * (l[0] + l[1]);
    o.s[1] = 0.5 * (h[0] + h[1]);
    o.d[0] = 0.5 * (l[1] - l[0]);
    o.d[1] = 0.5 * (h[1] - h[0]);
    o.r[0] = o.s[0] + s[0];
    o.r[1] = o.s[1] + s[1];
}

}  // namespace fx
}  // namespace gbr
