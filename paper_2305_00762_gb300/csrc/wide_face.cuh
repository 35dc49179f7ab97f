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
// shear velocity far below the stencil's: 2% of the faces of a developed
// four-quadrant flow, scattered over a sixth of its warps. What they cost is a
// chain of dependent instructions that the rest of the CTA waits for, so a warp
// takes its faces eight at a time, four lanes a face: a lane forms the functionals
// about one of the cells j-1 .. j+2, and then the limited value of one side. The
// code is kept out of line: inlined, its registers would be taken from every face.
// (One face a lane, gradients and differences in FP64 as well: four-quadrant 1024^2
// 4.18 ms a pass, double Mach 2.51; a lane a face with the functionals on integers
// 4.17 and 2.22; four lanes 4.13 and 2.11.)
//
// What the accuracy costs, us a pass without / with flags and this code: 64^2 vortex
// 880 / 908, four-quadrant 400^2 1450 / 1597, 1024^2 3983 / 4147, 4096^2 30770 /
// 32640, viscous 1280 x 640 3752 / 3877, MEG7-cons 400^2 1918 / 2389, double Mach
// 1024 x 256 (a shock of ratio 116 through four tiles a row) 1878 / 2114. The flags
// are 2.5% everywhere; a tile with a line of such faces takes 1.25 times as long.
//
// The MP test's absolute threshold, which fixed point leaves out, is applied here,
// and faces where it may tell (is_small_field) are evaluated here too: none in
// ordinary units; four-quadrant 1024^2 with densities of 1e-4 4.19 ms a pass, 1e-12
// 4.30, 1e-20 5.28.
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

// The four lanes of a face. V is a value of each; each(f) is f(k) of lane k,
// pick(x, k) lane k's value, own(x, k) the same where k is the lane itself.
#ifdef __CUDACC__
struct WideLanes {
    typedef double V;
    int base;  // the first one
    template <typename F>
    __device__ __forceinline__ V each(F f) const { return f((int)threadIdx.x & 3); }
    __device__ __forceinline__ double pick(const V& x, int k) const { return __shfl_sync(0xffffffffu, x, base + k); }
    __device__ __forceinline__ double own(const V& x, int) const { return x; }
};
#define GBR_LANES __device__ __forceinline__
#define GBR_LANES_CALL __device__ __noinline__
#else
struct WideLanes {
    struct V {
        double x[4];
    };
    template <typename F>
    V each(F f) const { return V{{f(0), f(1), f(2), f(3)}}; }
    double pick(const V& a, int k) const { return a.x[k]; }
    double own(const V& a, int k) const { return a.x[k]; }
};
#define GBR_LANES inline
#define GBR_LANES_CALL inline
#endif

// A variable or field about the cells j-1 .. j+2 (lane k: cell j-1+k): its value,
// the curvature functional d, and for k = 1, 2 the GRB functional n of the left
// and the right value (fixed_face.cuh).
struct WideField {
    WideLanes::V v, d, n;
};
template <int ORDER>
GBR_HD void wide_functionals(const Face& f, int variable, int k, double& v, double& d, double& n)
{
    const int at = f.at(variable) + (k - 1) * f.step;
    i64 q[9];
    int e[9], s = kExpMin;
#pragma unroll
    for (int c = 0; c < 9; ++c) {
        q[c] = f.m[at + (c - 4) * f.step];
        e[c] = f.e[at + (c - 4) * f.step];
        s = larger(s, e[c]);
    }
    v = unsplit(q[4], e[4]);
#pragma unroll
    for (int c = 0; c < 9; ++c) q[c] = aligned(q[c], e[c], s);
    const i64 c2 = q[4] + q[4];
    const i64 B1 = q[5] + q[3] - c2, B2 = c2 - q[6] - q[2];  // (B2, B4, A2 with their signs changed)
    const i64 B3 = q[7] + q[1] - c2, B4 = c2 - q[8] - q[0];
    const i64 A1 = q[5] - q[3], A2 = q[2] - q[6], A3 = q[7] - q[1];
    Acc curv, even, odd;
    curv.add(B1, 231);
    curv.add(B2, 44);
    curv.add(B3, 9);
    curv.add(B4, 1);
    if (ORDER == 4) {
        even.add(B1, 1617);
        even.add(B2, 308);
        even.add(B3, 63);
        even.add(B4, 7);
        odd.add(A1, 3780);
        odd.add(A2, 756);
        odd.add(A3, 84);
    } else {
        even.add(B1, 169);
        even.add(B2, 41);
        even.add(B3, 9);
        even.add(B4, 1);
        odd.add(A1, 315);
        odd.add(A2, 63);
        odd.add(A3, 7);
    }
    const Acc sum = k == 2 ? even - odd : even + odd;
    d = to_double(curv.shift<kCurvShift>(), s);
    n = to_double(sum.shift<ORDER == 4 ? kGrbShift4 : kGrbShift7>(), s);
}
template <int ORDER>
GBR_LANES WideField wide_variable(const WideLanes& L, const Face& f, int variable)
{
    WideField o;
#ifdef __CUDACC__
    wide_functionals<ORDER>(f, variable, (int)threadIdx.x & 3, o.v, o.d, o.n);
#else
    for (int k = 0; k < 4; ++k) wide_functionals<ORDER>(f, variable, k, o.v.x[k], o.d.x[k], o.n.x[k]);
#endif
    return o;
}
// x + a y
GBR_LANES WideField combine(const WideLanes& L, const WideField& x, double a, const WideField& y)
{
    WideField o;
    o.v = L.each([&](int k) { return fmadd(a, L.own(y.v, k), L.own(x.v, k)); });
    o.d = L.each([&](int k) { return fmadd(a, L.own(y.d, k), L.own(x.d, k)); });
    o.n = L.each([&](int k) { return fmadd(a, L.own(y.n, k), L.own(x.n, k)); });
    return o;
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

// The MEG7 values (Eqs. grb, mp5Condition, mp-procedure) of a field carried at
// `scale` times its value: the left one in lanes 0 and 2, the right one in 1 and 3.
template <int ORDER>
GBR_LANES WideLanes::V wide_limited(const WideLanes& L, const WideField& f, double scale)
{
    constexpr double kN = ORDER == 4 ? 8192.0 / 10080.0 : 1024.0 / 840.0, kD = 128.0 / 120.0;  // n, d -> delta, d_j
    const double st = 1e-20 * scale, thr = st * st;
    return L.each([&](int k) {
        const int s = k & 1;
        const double c = L.pick(f.v, 1 + s), o = L.pick(f.v, 2 - s), a = L.pick(f.v, 3 * s) - c;  // own cell, across, behind
        const double dc = L.pick(f.d, 1 + s), da = L.pick(f.d, 2 - s), db = L.pick(f.d, 3 * s);
        const double delta = kN * L.pick(f.n, 1 + s), m = minmod(o - c, -7.0 * a), v = c + delta;
        const double md = 0.5 * fmadd(-kD, minmod(dc, da), c + o), ul = fmadd(-7.0, a, c);
        const double lc = fmadd(4.0 / 3.0 * kD, minmod(dc, db), fmadd(-0.5, a, c));
        return delta * (delta - m) <= thr ? v : mp_clamp(c, o, md, ul, lc, v);
    });
}

// ut; and rho, un and p, of fields as in face_states: p -/+ rho c un and rho -
// p / c^2 (the sides in the lanes of wide_limited).
template <int ORDER>
GBR_LANES WideLanes::V wide_shear(const WideLanes& L, const Face& f)
{
    return wide_limited<ORDER>(L, wide_variable<ORDER>(L, f, 2), 1.0);
}
template <int ORDER>
GBR_LANES void wide_states(const WideLanes& L, const Face& f, double gamma, WideLanes::V& ro, WideLanes::V& uo, WideLanes::V& po)
{
    const WideField P = wide_variable<ORDER>(L, f, 3), R = wide_variable<ORDER>(L, f, 0);
    const double r = 0.5 * (L.pick(R.v, 1) + L.pick(R.v, 2)), gp = gamma * (0.5 * (L.pick(P.v, 1) + L.pick(P.v, 2)));
    const double y = rsqrt(gp * r), c = gp * y, rc = r * c, ic = r * y, ic2 = ic * ic;
    const WideLanes::V s = wide_limited<ORDER>(L, combine(L, R, -ic2, P), 1.0);
    const WideField U = wide_variable<ORDER>(L, f, 1);
    const WideLanes::V a = wide_limited<ORDER>(L, combine(L, P, -rc, U), 2.0 * c * c);
    const WideLanes::V b = wide_limited<ORDER>(L, combine(L, P, rc, U), 2.0 * c * c);
    ro = L.each([&](int k) { return fmadd(0.5 * ic2, L.own(a, k) + L.own(b, k), L.own(s, k)); });
    uo = L.each([&](int k) { return 0.5 * y * (L.own(b, k) - L.own(a, k)); });
    po = L.each([&](int k) { return 0.5 * (L.own(a, k) + L.own(b, k)); });
}

// MEG7-cons: w3, and the others of ConsStates. (Four variables and four fields: a
// call each, 400^2 pass 2465 -> 2402 us; for the primitive form's a call is slower
// than the copies, 1024^2 4131 -> 4157.)
template <int ORDER>
GBR_LANES_CALL WideField wide_variable_call(WideLanes L, Face f, int variable)
{
    return wide_variable<ORDER>(L, f, variable);
}
template <int ORDER>
GBR_LANES_CALL WideLanes::V wide_limited_call(WideLanes L, WideField f, double scale)
{
    return wide_limited<ORDER>(L, f, scale);
}
template <int ORDER>
GBR_LANES WideLanes::V wide_cons_shear(const WideLanes& L, const Face& f, double v)
{
    const WideField Q = wide_variable_call<ORDER>(L, f, 0), W = wide_variable_call<ORDER>(L, f, 2);
    return wide_limited_call<ORDER>(L, combine(L, W, -v, Q), 1.0);
}
template <int ORDER>
GBR_LANES void wide_cons_states(const WideLanes& L, const Face& f, const ConsCoefs& C, WideLanes::V& ro, WideLanes::V& so, WideLanes::V& uo)
{
    WideField zero, Q = wide_variable_call<ORDER>(L, f, 3);
    zero.v = zero.d = zero.n = L.each([](int) { return 0.0; });
    WideField A = combine(L, zero, C.b1, Q), T;  // A and t as in cons_states
    Q = wide_variable_call<ORDER>(L, f, 1);
    A = combine(L, A, -C.b1u, Q);
    T = combine(L, zero, -C.ic, Q);
    A = combine(L, A, -C.b1v, wide_variable_call<ORDER>(L, f, 2));
    Q = wide_variable_call<ORDER>(L, f, 0);
    A = combine(L, A, C.b2, Q);
    T = combine(L, T, C.uc, Q);
    const WideLanes::V a = wide_limited_call<ORDER>(L, combine(L, A, 1.0, T), 2.0);   // 2 w1
    const WideLanes::V b = wide_limited_call<ORDER>(L, combine(L, A, -1.0, T), 2.0);  // 2 w4
    const WideLanes::V c = wide_limited_call<ORDER>(L, combine(L, Q, -1.0, A), 1.0);  // w2
    so = L.each([&](int k) { return 0.5 * (L.own(a, k) + L.own(b, k)); });
    uo = L.each([&](int k) { return 0.5 * (L.own(b, k) - L.own(a, k)); });
    ro = L.each([&](int k) { return L.own(so, k) + L.own(c, k); });
}

#ifdef __CUDACC__
// The faces of a warp that are flagged, by the whole warp: work(L, src) with the
// lanes L of a face and the lane src it belongs to (a group without one repeats
// the first), then take(from) with the lane that holds the left values of this
// lane's face (the next one holds the right ones), or -1.
template <typename W, typename T>
__device__ __forceinline__ void wide_faces(bool wide, W work, T take)
{
    const int lane = (int)threadIdx.x & 31;
    unsigned todo = __ballot_sync(0xffffffffu, wide);
    while (todo) {
        unsigned rest = todo;
        int src = __ffs((int)todo) - 1;
#pragma unroll
        for (int g = 0; g < 8; ++g) {
            if (g == lane >> 2 && rest) src = __ffs((int)rest) - 1;
            rest &= rest - 1u;
        }
        work(WideLanes{lane & 28}, src);
        const int rank = __popc(todo & ((1u << lane) - 1u));
        take(((todo >> lane) & 1u) && rank < 8 ? 4 * rank : -1);
        todo = rest;
    }
}
// Lane `from`'s x (the left value) and the next one's, where from >= 0.
__device__ __forceinline__ void wide_take(double x, int from, double (&o)[2])
{
    const double l = __shfl_sync(0xffffffffu, x, from & 31), r = __shfl_sync(0xffffffffu, x, (from + 1) & 31);
    if (from >= 0) {
        o[0] = l;
        o[1] = r;
    }
}
// The planes and the face of each lane: the cell before it and its direction.
struct WideFace {
    const i64* m;
    const unsigned short* e;
    int values, row;  // values per plane; distance of rows
    int cell;
    bool x;
    __device__ __forceinline__ Face of(int src) const
    {
        const int c = __shfl_sync(0xffffffffu, 2 * cell + (x ? 1 : 0), src);
        return Face{m + (c >> 1), e + (c >> 1), c & 1 ? 1 : row, values, c & 1 ? 1 : 2};
    }
};
template <int ORDER>
__device__ __noinline__ void wide_shear_warp(WideFace f, bool wide, double (&ut)[2])
{
    double u;
    wide_faces(
        wide, [&](const WideLanes& L, int src) { u = wide_shear<ORDER>(L, f.of(src)); }, [&](int from) { wide_take(u, from, ut); });
}
template <int ORDER>
__device__ __noinline__ void wide_states_warp(WideFace f, bool wide, double gamma, FaceStates& o)
{
    double r, u, p;
    wide_faces(
        wide, [&](const WideLanes& L, int src) { wide_states<ORDER>(L, f.of(src), gamma, r, u, p); },
        [&](int from) {
            wide_take(r, from, o.r);
            wide_take(u, from, o.un);
            wide_take(p, from, o.p);
        });
}
template <int ORDER>
__device__ __noinline__ void wide_cons_shear_warp(WideFace f, bool wide, double v, double (&w3)[2])
{
    double w;
    wide_faces(
        wide, [&](const WideLanes& L, int src) { w = wide_cons_shear<ORDER>(L, f.of(src), __shfl_sync(0xffffffffu, v, src)); },
        [&](int from) { wide_take(w, from, w3); });
}
template <int ORDER>
__device__ __noinline__ void wide_cons_states_warp(WideFace f, bool wide, ConsCoefs C, ConsStates& o)
{
    double r, s, d;
    wide_faces(
        wide,
        [&](const WideLanes& L, int src) {
            auto of = [&](double x) { return __shfl_sync(0xffffffffu, x, src); };
            ConsCoefs S;
            S.b1 = of(C.b1);
            S.b1u = of(C.b1u);
            S.b1v = of(C.b1v);
            S.b2 = of(C.b2);
            S.uc = of(C.uc);
            S.ic = of(C.ic);
            S.v = of(C.v);
            wide_cons_states<ORDER>(L, f.of(src), S, r, s, d);
        },
        [&](int from) {
            wide_take(r, from, o.r);
            wide_take(s, from, o.s);
            wide_take(d, from, o.d);
        });
}
#endif

}  // namespace fx
}  // namespace gbr
