// MEG7-prim face states in 64-bit fixed point (the FP64 form's characteristic
// reconstruction on the integer pipe).
//
// GB300 issues one FP64 warp instruction per 19 clocks and SM, where a 64-bit
// integer add takes one clock and a 64 x 64 -> high 64 product about five, and
// the two run side by side. Everything between the staged primitives and the
// face states (gradients, GRB sums, characteristic projection, MP limiter) is
// linear or a comparison, so it is done here on integers, exactly up to the
// rounding of the projection products.
//
// Measured, FP64 step of three stages: with FP64 arithmetic throughout (the FP64
// pipe saturated) 1024^2 6.57 ms, 400^2 1.28 ms, viscous 1280 x 640 6.06 ms;
// with the face states here 3.66 / 0.73 / 3.93 ms; with the roots and
// reciprocals, the primitives, the cell fluxes and their reconstruction on
// integers too (fixed_math.cuh, fixed_stage.cuh) 1.99 / 0.36 / 1.88 ms, and
// 2.08 / 0.40 / 1.94 ms with the faces beside strong jumps at the accuracy of their
// own cells (wide_face.cuh). The stage is then bound by the integer pipe and FP64
// about alike (57% and 61% of what each can issue), at 16 warps an SM.
//
// Scaling. A variable q of one face's stencil (cells j-5 .. j+6) is held as
// I = q / 2^(e - 1081) with e the largest biased exponent of the stencil, so
// |I| < 2^kBits: values within 2^6 of the largest are held exactly, smaller
// ones rounded down at 2^-59 of it. The scale depends on the face's own stencil
// only: the result does not depend on tiles, slabs or batches. The limiter
// bounds a state by the cells beside the face, which may be far smaller than the
// largest value: such faces are flagged (kWide) and evaluated by wide_face.cuh.
// Error of a state in units of 2^-53 of its own cell's terms, root mean square
// over jumps of every kind (and of the same formulas in FP64 throughout): rho
// 0.1 - 0.5 (0.3 - 0.5), un 0.1 - 0.5 (0.4 - 0.5), p 0.1 - 0.4 (0.4 - 0.5);
// MEG7-cons at Mach numbers up to 3 rho 0.7 - 1.3 (0.9 - 1.4), un 0.2 - 0.5
// (0.4 - 0.6), p 1.3 - 2.5 (1.9 - 2.9).
//
// Linear functionals. The left value at j+1/2 and the curvatures of the MP
// limiter are sums over the even and odd differences about a cell,
// B_k = q_{+k} + q_{-k} - 2 q_0 and A_k = q_{+k} - q_{-k}; with the
// sixth-order gradients of Eq. six put into Eq. grb and into d_j,
//   840 (Phi^L_j - Phi_j) = 169 B1 - 41 B2 + 9 B3 - B4 + 315 A1 - 63 A2 + 7 A3,
//   120 d_j               = 231 B1 - 44 B2 + 9 B3 - B4,
// and the right value about cell j+1 takes the odd part with its sign
// changed. They are formed once per variable and then projected (ten
// functionals per variable instead of six values and six gradients).
//
// The MP test (Eq. mp5Condition, (Phi^L - Phi_j)(Phi^L - Phi^MP) <= 1e-40) is
// not taken: where the product is not positive, Phi^L lies between Phi_j and
// Phi^MP, so inside both intervals of Eq. mp-procedure, and the clamp to
// [Phi^min, Phi^max] returns it unchanged; on integers this holds exactly. A
// positive product up to 1e-40 moves the result by at most 1e-20. Where that is
// more than rounding (fields below about 2^-12), faces with a limited value that
// close to its unlimited one are evaluated with the test (is_small_field).
//
// Overflow. With |I| < 2^59 = M after projection the largest intermediate is
// the bound UL = Phi_j + 7 (Phi_j - Phi_{j-1}), at most 15 M < 2^63 (LC: 14.7 M).
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define GBR_HD __host__ __device__ __forceinline__
#define GBR_CALL __host__ __device__ __noinline__
#else
#define GBR_HD inline
#define GBR_CALL inline
#include <string.h>
#endif

namespace gbr {
namespace fx {

typedef long long i64;
typedef unsigned long long u64;

constexpr int kBits = 59;           // |I| < 2^kBits
constexpr int kExpMin = 128;        // smaller stencils count as zero
constexpr int kExpMax = 1900;       // larger ones (infinities, NaN included) are refused
constexpr int kOne = 1022 + kBits;  // I of a stencil with exponent e has units 2^(e - kOne)

GBR_HD u64 bits_of(double x)
{
#ifdef __CUDA_ARCH__
    return (u64)__double_as_longlong(x);
#else
    u64 u;
    memcpy(&u, &x, 8);
    return u;
#endif
}
GBR_HD double of_bits(u64 u)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((i64)u);
#else
    double x;
    memcpy(&x, &u, 8);
    return x;
#endif
}
GBR_HD u64 mulhi_u(u64 a, u64 b)
{
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (u64)(((unsigned __int128)a * b) >> 64);
#endif
}
// x r / 2^64, x signed, r < 2^63, within three units: three 32 x 32 -> 64
// products (the low halves' product and the lowest bits of r's halves are
// dropped) instead of four and the sign's correction. The addend, nearly a unit,
// centres the error of what is dropped; zero stays zero.
GBR_HD i64 mulhi(i64 x, u64 r)
{
    const int xh = (int)(x >> 32), rh = (int)(r >> 32);
    const i64 mid = 0x7fffffffll + (i64)xh * (int)((unsigned)r >> 1) + (i64)((u64)(unsigned)x * ((unsigned)rh >> 1));
    return (i64)xh * rh + (mid >> 31);
}

GBR_HD int larger(int a, int b) { return a > b ? a : b; }
GBR_HD int exponent(double x) { return (int)(bits_of(x) >> 52) & 0x7ff; }

// A value taken apart once, where it is produced, so that each of the many
// stencils that read it only shifts: x = m 2^(e - kOne), |m| < 2^kBits. For a
// double, e is its biased exponent (zeros and subnormals: m = 0, e = 1).
GBR_HD void split(double x, i64& m, unsigned short& e)
{
    const u64 b = bits_of(x);
    const int ex = (int)(b >> 52) & 0x7ff;
    const i64 v = (i64)(((b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull) << (kBits - 53)), g = (i64)b >> 63;
    m = ex == 0 ? 0 : (v ^ g) - g;
    e = (unsigned short)(ex == 0 ? 1 : ex);
}
// The split value m, ex in units 2^(e - kOne), ex <= e, rounded down.
GBR_HD i64 aligned(i64 m, int ex, int e)
{
#ifdef __CUDA_ARCH__
    i64 r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(m), "r"(e - ex));  // (a shift past the width counts as the width)
    return r;
#else
    const int s = e - ex;
    return m >> (s < 63 ? s : 63);
#endif
}

// x 2^(e - kOne) as a double, rounded to nearest; kExpMin <= e <= kExpMax + 64.
GBR_HD double to_double(i64 x, int e)
{
    const i64 g = x >> 63;
    const u64 u = (u64)((x ^ g) - g);
    unsigned h = (unsigned)(u >> 32), l = (unsigned)u;
    int n = 0;
    if (h == 0) {
        h = l;
        l = 0;
        n = 32;
    }
#ifdef __CUDA_ARCH__
    const int z = __clz((int)h);
    h = __funnelshift_l(l, h, z);
#else
    const int z = h ? __builtin_clz(h) : 32;
    h = z == 0 ? h : (z == 32 ? 0u : (h << z) | (l >> (32 - z)));
#endif
    l = z == 32 ? 0u : l << z;
    n += z;
    const u64 t = ((u64)h << 32) | l;
    u64 r = ((u64)(unsigned)(e + 63 - kBits - n) << 52) + (t >> 11) + ((t >> 10) & 1u);
    r |= (u64)g & 0x8000000000000000ull;
    return of_bits(h == 0 ? 0ull : r);
}

// The double nearest to a split value.
GBR_HD double unsplit(i64 m, int e)
{
    const double x = to_double(m, e < kExpMin ? kExpMin : e);
    return e < kExpMin ? 0.0 : e <= kExpMax ? x : of_bits(0x7ff8000000000000ull);
}

// Sum of c X over a few X (|X| < 2^62) and small positive integers c, exact.
struct Acc {
    i64 hi;
    u64 lo;
    GBR_HD Acc() : hi(0), lo(0) {}
    GBR_HD void add(i64 x, unsigned c)
    {
        hi += (i64)(int)(x >> 32) * (int)c;
        lo += (u64)(unsigned)x * c;
    }
    GBR_HD Acc operator+(const Acc& o) const
    {
        Acc r;
        r.hi = hi + o.hi;
        r.lo = lo + o.lo;
        return r;
    }
    GBR_HD Acc operator-(const Acc& o) const
    {
        Acc r;
        r.hi = hi - o.hi;
        r.lo = lo - o.lo;  // (signed from here on)
        return r;
    }
    template <int S>
    GBR_HD i64 shift() const { return hi * (1ll << (32 - S)) + ((i64)lo >> S); }  // floor(sum / 2^S)
};

// Fixed-point factors: round(num / den 2^64) for num < den.
constexpr u64 ratio(u64 num, u64 den)
{
    u64 q = 0, r = num;
    for (int i = 0; i < 64; ++i) {
        r *= 2;
        q = 2 * q + (r >= den ? 1 : 0);
        if (r >= den) r -= den;
    }
    return q + (2 * r >= den ? 1 : 0);
}

// The functionals of one variable at one face: its values at cells j-1..j+2,
// the GRB corrections of the left value (about cell j) and the right one
// (about j+1), and the curvatures d_{j-1} .. d_{j+2}; corrections and
// curvatures scaled by kGrb<ORDER> and kCurv.
struct Functionals {
    i64 v[4], n[2], d[4];
};
constexpr int kGrbShift7 = 10;  // n = 840 delta / 2^10
constexpr int kGrbShift4 = 13;  // order 4: n = 10080 delta / 2^13
constexpr int kCurvShift = 7;   // d = 120 d_j / 2^7

template <int ORDER>
GBR_HD void functionals(const i64 (&q)[12], Functionals& f)
{
#pragma unroll
    for (int k = 0; k < 4; ++k) f.v[k] = q[4 + k];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int c = 4 + k;
        const i64 c2 = q[c] + q[c];
        const i64 B1 = q[c + 1] + q[c - 1] - c2, B2 = c2 - q[c + 2] - q[c - 2];  // (B2, B4, A2 with their signs changed)
        const i64 B3 = q[c + 3] + q[c - 3] - c2, B4 = c2 - q[c + 4] - q[c - 4];
        Acc d;
        if (ORDER == 4 || k == 0 || k == 3) {
            d.add(B1, 231);
            d.add(B2, 44);
            d.add(B3, 9);
            d.add(B4, 1);
        }
        if (k == 1 || k == 2) {
            const i64 A1 = q[c + 1] - q[c - 1], A2 = q[c - 2] - q[c + 2], A3 = q[c + 3] - q[c - 3];
            Acc even, odd;
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
                d = even;
                d.add(B1, 62);
                d.add(B2, 3);
            }
            const Acc n = k == 1 ? even + odd : even - odd;
            f.n[k - 1] = n.shift<ORDER == 4 ? kGrbShift4 : kGrbShift7>();
        }
        f.d[k] = d.shift<kCurvShift>();
    }
}

// f r / 2^64 of every functional.
GBR_HD void scale(const Functionals& f, u64 r, Functionals& o)
{
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        o.v[k] = mulhi(f.v[k], r);
        o.d[k] = mulhi(f.d[k], r);
    }
    o.n[0] = mulhi(f.n[0], r);
    o.n[1] = mulhi(f.n[1], r);
}
GBR_HD void sum(const Functionals& a, const Functionals& b, Functionals& o)
{
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        o.v[k] = a.v[k] + b.v[k];
        o.d[k] = a.d[k] + b.d[k];
    }
    o.n[0] = a.n[0] + b.n[0];
    o.n[1] = a.n[1] + b.n[1];
}
GBR_HD void difference(const Functionals& a, const Functionals& b, Functionals& o)
{
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        o.v[k] = a.v[k] - b.v[k];
        o.d[k] = a.d[k] - b.d[k];
    }
    o.n[0] = a.n[0] - b.n[0];
    o.n[1] = a.n[1] - b.n[1];
}

// Every functional / 2^k: from a finer scale to one k larger.
GBR_HD void shift_right(Functionals& f, int k)
{
    k = k < 63 ? k : 63;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        f.v[i] >>= k;
        f.d[i] >>= k;
    }
    f.n[0] >>= k;
    f.n[1] >>= k;
}

// Eq. alpha's minmod.
GBR_HD i64 minmod(i64 a, i64 b)
{
    const bool first = (a < b) != (a < 0);  // same signs: the smaller magnitude
    const i64 r = first ? a : b;
    return (a ^ b) < 0 ? 0 : r;
}

// pl clamped to [Phi^min, Phi^max] of Eq. mp-procedure (min distributes over
// max: four comparisons a bound instead of five).
GBR_HD i64 mp_clamp(i64 p2, i64 p3, i64 md, i64 ul, i64 lc, i64 pl)
{
    const bool c1 = p3 < md, c2 = ul < lc;
    const i64 n1 = c1 ? p3 : md, x1 = c1 ? md : p3;
    const i64 n2 = c2 ? ul : lc, x2 = c2 ? lc : ul;
    const i64 n3 = n1 > n2 ? n1 : n2, x3 = x1 < x2 ? x1 : x2;
    const i64 mn = p2 < n3 ? p2 : n3, mx = p2 > x3 ? p2 : x3;
    const i64 r = pl > mn ? pl : mn;
    return r < mx ? r : mx;
}

// n -> delta = Phi^GRB - Phi_j: 2^10 / 840 = 1 + 184/840; 2^13 / 10080 = 1 - 1888/10080.
template <int ORDER>
GBR_HD i64 grb_delta(i64 n)
{
    return ORDER == 4 ? n - mulhi(n, ratio(1888, 10080)) : n + mulhi(n, ratio(184, 840));
}

// The MP-limited left and right values (Eqs. grb, mp-procedure) at the face.
template <int ORDER>
GBR_HD void limited(const Functionals& f, i64& vl, i64& vr)
{
    const i64 aL = f.v[0] - f.v[1], aR = f.v[3] - f.v[2];
    const i64 mc = minmod(f.d[1], f.d[2]), mL = minmod(f.d[1], f.d[0]), mR = minmod(f.d[2], f.d[3]);
    // d = 120 d_j / 128: d_j = d + d 8/120, 4/3 d_j = d + d (512 - 360)/360
    const i64 md = (f.v[1] + f.v[2] - mc - mulhi(mc, ratio(8, 120))) >> 1;
    const i64 lcL = f.v[1] - (aL >> 1) + mL + mulhi(mL, ratio(152, 360));
    const i64 lcR = f.v[2] - (aR >> 1) + mR + mulhi(mR, ratio(152, 360));
    vl = mp_clamp(f.v[1], f.v[2], md, f.v[1] - 7 * aL, lcL, f.v[1] + grb_delta<ORDER>(f.n[0]));
    vr = mp_clamp(f.v[2], f.v[1], md, f.v[2] - 7 * aR, lcR, f.v[2] + grb_delta<ORDER>(f.n[1]));
}

// Twelve split values of one variable, cells j-5 .. j+6, and their scale.
struct Stencil {
    i64 m[12];
    int e[12];
};
GBR_HD int stencil_exponent(const Stencil& x)
{
    int e = kExpMin;
#pragma unroll
    for (int k = 0; k < 12; ++k) e = x.e[k] > e ? x.e[k] : e;
    return e;
}

template <int ORDER>
GBR_HD void variable(const Stencil& x, int e, Functionals& f)
{
    i64 q[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) q[k] = aligned(x.m[k], x.e[k], e);
    functionals<ORDER>(q, f);
}

// A positive number m / 2^63 2^(e - 1023), 2^63 <= m < 2^64, e a biased exponent
// that may run outside a double's range. Products are rounded down in the last
// of 63 bits.
struct Pos {
    u64 m;
    int e;
};

// A factor a applied to a variable of scale e, for a result of scale eo: the r
// of scale(). The product's own scale is e + a.e - 1022, and eo is at least that.
GBR_HD u64 factor(const Pos& a, int e, int eo)
{
    const int k = eo - (e + a.e - 1022);
    return k < 63 ? a.m >> k : 0;
}
GBR_HD u64 factor(double a, int e, int eo)  // of |a|
{
    Pos p;
    p.m = (bits_of(a) << 11) | 0x8000000000000000ull;
    p.e = exponent(a);
    return factor(p, e, eo);
}

// Faces whose states fixed point would hold with fewer bits than FP64 arithmetic
// does (wide_face.cuh evaluates them): the scale of the stencil exceeds the
// largest term of a cell beside the face by more than kWide binary orders. A
// result carries a few units of 2^-59 of the scale, so up to there its error is
// a few units of 2^(kWide-59) of its own terms.
constexpr int kWide = 5;
GBR_HD bool is_wide(int scale, int local0, int local1) { return scale - (local0 < local1 ? local0 : local1) > kWide; }
// Nor are faces where the MP test's threshold may tell: a value it leaves unlimited
// lies within 1e-20 (2^-66.4) of the limiter's, times 2^k where the field is carried
// at up to 2^k times its value. Asked where that is 2^-55 or more of the scale.
constexpr int kSmall = kOne - 70;
GBR_HD bool is_small(int scale, int k) { return scale - k <= kSmall; }
GBR_HD bool within(i64 d, int bits)
{
    const i64 g = d >> 63;
    return d != 0 && ((d ^ g) >> (bits < 62 ? bits : 62)) == 0;
}
// (a call, so that other faces branch past it)
template <int ORDER>
GBR_CALL bool small_tells(i64 cl, i64 nl, i64 l, i64 cr, i64 nr, i64 r, int bits)
{
    return within(cl + grb_delta<ORDER>(nl) - l, bits) || within(cr + grb_delta<ORDER>(nr) - r, bits);
}
template <int ORDER>
GBR_HD bool is_small_field(const Functionals& f, i64 l, i64 r, int scale, int k)
{
    bool s = false;
    if (is_small(scale, k)) s = small_tells<ORDER>(f.v[1], f.n[0], l, f.v[2], f.n[1], r, kOne - 66 - scale + k);
    return s;
}
// The same from a field's values (l, r): a value, its step from the cell's value
// and the cell's other terms (tl, tr) all below 2^-kWide of the scale. (A field
// may be small at one cell, as where a velocity changes sign, without losing
// anything: FP64 rounds its step too, and an unlimited value carries the
// rounding of the differences that it was formed of.)
GBR_HD unsigned leading(i64 x) { return (unsigned)((int)(x >> 32) ^ (int)(x >> 63)); }
template <int ORDER>
GBR_HD bool is_wide_field(const Functionals& f, i64 l, i64 r, i64 tl = 0, i64 tr = 0)
{
    const i64 al = l == f.v[1] + grb_delta<ORDER>(f.n[0]) ? f.v[2] - f.v[0] : 0;
    const i64 ar = r == f.v[2] + grb_delta<ORDER>(f.n[1]) ? f.v[3] - f.v[1] : 0;
    const unsigned L = leading(f.v[1]) | leading(l - f.v[1]) | leading(al) | leading(tl);
    const unsigned R = leading(f.v[2]) | leading(r - f.v[2]) | leading(ar) | leading(tr);
    return (L < R ? L : R) >> (kBits - kWide - 32) == 0;
}

// The face states (L, R) back in primitives.
struct FaceStates {
    double r[2], un[2], ut[2], p[2];
    bool ok;    // false: a stencil value too large, infinite or NaN
    bool wide;  // r, un, p: to be evaluated in FP64
    bool wide_ut;
};

// A shear velocity below 2^-kStill of the speed of sound throughout the stencil is
// rounding noise or as good as none, and stays in fixed point: its error is then
// below 2^(-59-kStill) of a speed of sound that the normal velocity is rounded at
// 2^-53 of. The exponent of that bound from the speed's (the cells': c^2 ~ p / rho).
// Nor is the MP test's 1e-20 taken into account for a shear velocity unless it
// exceeds what the speed of sound is rounded at; then nothing is still either.
constexpr int kStill = 20;
GBR_HD int still_exponent(int c) { return c <= kSmall + 5 ? kExpMin : larger(c - kStill, kExpMin); }
GBR_HD int still_exponent(int r0, int p0, int r1, int p1)
{
    return still_exponent(1023 + ((p0 - r0 < p1 - r1 ? p0 - r0 : p1 - r1) >> 1));
}

// Field 3 (shear) is ut itself. Returns whether its stencil is in range.
template <int ORDER, typename F>
GBR_HD bool shear_states(F load, int still, double (&ut)[2], bool& wide)
{
    Stencil x;
    load(2, x);
    const int e = stencil_exponent(x);
    Functionals R;
    variable<ORDER>(x, e, R);
    i64 l, r;
    limited<ORDER>(R, l, r);
    ut[0] = to_double(l, e);
    ut[1] = to_double(r, e);
    wide = e > still && ((still == kExpMin && is_small_field<ORDER>(R, l, r, e, 0)) || (is_wide(e + 1, x.e[5], x.e[6]) && is_wide_field<ORDER>(R, l, r)));
    return e <= kExpMax;
}

// The other three, and the states (SHEAR: ut too).
// load(m, x): the stencil of variable m (0 rho, 1 un, 2 ut, 3 p); of the face's
// mean state, y = 1 / (2 rho c), rc2 = 2 rho c and ic2 = 1 / c^2. Fields: entropy
// w2 = rho - p / c^2; w1, w4 = p -/+ rho c un; shear w3 = ut. Back: p =
// (w1 + w4) / 2, un = (w4 - w1) y, rho = w2 + p / c^2.
template <int ORDER, bool SHEAR = true, typename F>
GBR_HD void face_states(F load, const Pos& y, const Pos& rc2, const Pos& ic2, FaceStates& o)
{
    Functionals P;
    i64 sl, sr;
    int ep, es, ew, lp[2], lr[2];  // lp, lr: of the cells beside the face
    {
        Stencil x;
        load(3, x);
        lp[0] = x.e[5];
        lp[1] = x.e[6];
        ep = stencil_exponent(x);
        variable<ORDER>(x, ep, P);
    }
    {  // field 2 (entropy): rho - p / c^2
        Stencil x;
        load(0, x);
        const int er = stencil_exponent(x), eprod = ep + ic2.e - 1022;
        es = (er > eprod ? er : eprod) + 1;
        lr[0] = x.e[5];
        lr[1] = x.e[6];
        o.wide = is_wide(es, larger(lr[0], lp[0] + ic2.e - 1022), larger(lr[1], lp[1] + ic2.e - 1022));
        Functionals R, S;
        scale(P, factor(ic2, ep, es), S);
        variable<ORDER>(x, es, R);
        difference(R, S, R);
        limited<ORDER>(R, sl, sr);
        o.wide = o.wide || is_small_field<ORDER>(R, sl, sr, es, 0);
    }
    {  // fields 1 and 4 (u -/+ c), carried as p -/+ rho c un
        Stencil x;
        load(1, x);
        const int eu = stencil_exponent(x), eprod = eu - 1 + rc2.e - 1022;  // (half of rc2)
        ew = (ep > eprod ? ep : eprod) + 1;
        o.wide = o.wide || is_wide(ew, larger(lp[0], x.e[5] + rc2.e - 1023), larger(lp[1], x.e[6] + rc2.e - 1023));
        Functionals U, W;
        variable<ORDER>(x, eu, U);
        scale(U, factor(rc2, eu - 1, ew), U);
        shift_right(P, ew - ep);
        i64 ml, mr, pl, pr;
        difference(P, U, W);
        limited<ORDER>(W, ml, mr);
        o.wide = o.wide || is_small_field<ORDER>(W, ml, mr, ew, 1024 - ic2.e);  // (carried at 2 c^2 times the paper's)
        sum(P, U, W);
        limited<ORDER>(W, pl, pr);
        o.wide = o.wide || is_small_field<ORDER>(W, pl, pr, ew, 1024 - ic2.e);
        const int ev = ew + y.e - 1021;  // (half the mantissa: a bit to spare)
        const bool some = ev >= kExpMin;  // smaller velocities count as zero
        o.un[0] = to_double(some ? mulhi(pl - ml, y.m >> 1) : 0, some ? ev : kExpMin);
        o.un[1] = to_double(some ? mulhi(pr - mr, y.m >> 1) : 0, some ? ev : kExpMin);
        pl += ml;  // 2 p: p in units one exponent lower
        pr += mr;
        o.p[0] = to_double(pl, ew - 1);
        o.p[1] = to_double(pr, ew - 1);
        const int eprod2 = ew - 1 + ic2.e - 1022, er = (es > eprod2 ? es : eprod2) + 1;
        const u64 fi = factor(ic2, ew - 1, er);
        o.r[0] = to_double(aligned(sl, es, er) + mulhi(pl, fi), er);
        o.r[1] = to_double(aligned(sr, es, er) + mulhi(pr, fi), er);
        o.ok = er <= kExpMax && ev <= kExpMax;
    }
    bool in_range = true;
    if constexpr (SHEAR) in_range = shear_states<ORDER>(load, still_exponent(lr[0], lp[0], lr[1], lp[1]), o.ut, o.wide_ut);
    o.ok = o.ok && ew <= kExpMax && es <= kExpMax && in_range;
}

// MEG7-cons: the reconstructed variables are rho, rho un, rho ut, E, projected
// with the left eigenvectors of the conservative flux Jacobian at the mean
// state. With A = b2 q0 - b1 (u q1 + v q2 - q3), b1 = (gamma - 1) / c^2, b2 =
// b1 (u^2 + v^2) / 2 and t = (u q0 - q1) / c the fields are w1 = (A + t) / 2,
// w2 = q0 - A, w3 = q2 - v q0, w4 = (A - t) / 2. The face state is returned as
// sums: rho = w1 + w2 + w4, s = w1 + w4, d = w4 - w1, w3.
struct ConsCoefs {
    double b1, b1u, b1v, b2, uc, ic, v;  // b1, b1 u, b1 v, b2, u / c, 1 / c, v
};
struct ConsStates {
    double r[2], s[2], d[2], w3[2];
    bool ok;    // false: a stencil value too large, infinite or NaN
    bool wide, wide_w3;  // r, s, d and w3: to be evaluated in FP64 (wide_face.cuh)
};

// acc += a f (acc -= with `minus`), a of any sign, r the factor() of |a|.
GBR_HD void accumulate(Functionals& acc, const Functionals& f, double a, u64 r, bool minus)
{
    const i64 g = (bits_of(a) >> 63) != (minus ? 1u : 0u) ? -1 : 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        acc.v[k] += (mulhi(f.v[k], r) ^ g) - g;
        acc.d[k] += (mulhi(f.d[k], r) ^ g) - g;
    }
    acc.n[0] += (mulhi(f.n[0], r) ^ g) - g;
    acc.n[1] += (mulhi(f.n[1], r) ^ g) - g;
}
// load(m, x): the stencil of variable m; scale(m): its stencil's exponent.
template <int ORDER, typename F, typename E>
GBR_HD void cons_states(F load, E scale_of, const ConsCoefs& C, ConsStates& o)
{
    int e[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) e[m] = scale_of(m);
    auto product = [](int es, double a) { return es + exponent(a) - 1022; };
    // A and t are sums of four and two terms, 2 w1 = A + t of six: three bits
    int ea = larger(larger(product(e[0], C.b2), product(e[1], C.b1u)), larger(product(e[2], C.b1v), product(e[3], C.b1)));
    ea = larger(ea, larger(product(e[0], C.uc), product(e[1], C.ic))) + 3;
    ea = larger(ea, kExpMin);
    const int es = larger(e[2], product(e[0], C.v)) + 1, er = larger(e[0], ea) + 1;
    int ql[2], la[2];  // exponents of q0, and of the terms of A and t, at the cells beside the face
    Functionals Q0, A, T, W;
    i64 tl, tr;
    {
        Stencil x;
        load(0, x);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            ql[k] = x.e[5 + k];
            la[k] = larger(product(ql[k], C.b2), product(ql[k], C.uc));
        }
        variable<ORDER>(x, e[0], Q0);
        scale(Q0, factor(C.b2, e[0], ea), A);
        const i64 g = (i64)bits_of(C.uc) >> 63;
        scale(Q0, factor(C.uc, e[0], ea), T);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            T.v[k] = (T.v[k] ^ g) - g;
            T.d[k] = (T.d[k] ^ g) - g;
        }
        T.n[0] = (T.n[0] ^ g) - g;
        T.n[1] = (T.n[1] ^ g) - g;
    }
    {
        Stencil x;
        Functionals Q;
        load(1, x);
#pragma unroll
        for (int k = 0; k < 2; ++k) la[k] = larger(la[k], larger(product(x.e[5 + k], C.b1u), product(x.e[5 + k], C.ic)));
        variable<ORDER>(x, e[1], Q);
        accumulate(A, Q, C.b1u, factor(C.b1u, e[1], ea), true);
        accumulate(T, Q, C.ic, factor(C.ic, e[1], ea), true);
        load(3, x);
#pragma unroll
        for (int k = 0; k < 2; ++k) la[k] = larger(la[k], product(x.e[5 + k], C.b1));
        variable<ORDER>(x, e[3], Q);
        accumulate(A, Q, C.b1, factor(C.b1, e[3], ea), false);
        load(2, x);
        variable<ORDER>(x, e[2], Q);
        accumulate(A, Q, C.b1v, factor(C.b1v, e[2], ea), true);
        W = Q;
        shift_right(W, es - e[2]);
        const i64 t0 = W.v[1], t1 = W.v[2];
        const int still = still_exponent((ql[0] < ql[1] ? ql[0] : ql[1]) + 1023 - exponent(C.ic));  // (momenta: rho c)
        accumulate(W, Q0, C.v, factor(C.v, e[0], es), true);
        limited<ORDER>(W, tl, tr);
        o.wide = is_wide(ea, la[0], la[1]) || is_wide(er, larger(ql[0], la[0]), larger(ql[1], la[1]));
        o.wide_w3 = es > still + 1 && ((still == kExpMin && is_small_field<ORDER>(W, tl, tr, es, 0)) || is_wide_field<ORDER>(W, tl, tr, t0, t1));
    }
    i64 al, ar, bl, br, cl, cr;  // 2 w1, 2 w4, w2
    sum(A, T, W);
    limited<ORDER>(W, al, ar);
    o.wide = o.wide || is_small_field<ORDER>(W, al, ar, ea, 1);
    difference(A, T, W);
    limited<ORDER>(W, bl, br);
    o.wide = o.wide || is_small_field<ORDER>(W, bl, br, ea, 1);
    shift_right(Q0, er - e[0]);
    shift_right(A, er - ea);
    difference(Q0, A, W);
    limited<ORDER>(W, cl, cr);
    o.wide = o.wide || is_small_field<ORDER>(W, cl, cr, er, 0);
    o.s[0] = to_double(al + bl, ea - 1);
    o.s[1] = to_double(ar + br, ea - 1);
    o.d[0] = to_double(bl - al, ea - 1);
    o.d[1] = to_double(br - ar, ea - 1);
    o.w3[0] = to_double(tl, es);
    o.w3[1] = to_double(tr, es);
    const int k = er + 1 - ea < 63 ? er + 1 - ea : 63;  // (al + bl is twice w1 + w4: one exponent lower)
    o.r[0] = to_double(cl + ((al + bl) >> k), er);
    o.r[1] = to_double(cr + ((ar + br) >> k), er);
    o.ok = ea <= kExpMax && es <= kExpMax && er <= kExpMax && e[3] <= kExpMax;
}

// 1/2 (F(f_L) + F(f_R)) at the face after cell j of one flux component, the
// symmetric 10-point stencil of Eq. flux-full and its mirror over split values
// at cells j-4 .. j+5 (weights / 1680; order 4: Eq. fourth, / 2880), exact up to
// the alignment of the values (2^-58 of the largest) and the final rounding.
template <int ORDER>
GBR_HD double recon_mean(const i64 (&m)[10], const int (&ex)[10])
{
    int e = kExpMin;
#pragma unroll
    for (int k = 0; k < 10; ++k) e = ex[k] > e ? ex[k] : e;
    i64 q[10];
#pragma unroll
    for (int k = 0; k < 10; ++k) q[k] = aligned(m[k], ex[k], e);
    Acc a;
    a.add(q[4] + q[5], ORDER == 4 ? 1821 : 1052);
    a.add(-q[3] - q[6], ORDER == 4 ? 461 : 250);
    a.add(q[2] + q[7], ORDER == 4 ? 85 : 38);
    if (ORDER == 4) {
        a.add(-q[1] - q[8], 4);
        a.add(-q[0] - q[9], 1);
    } else {
        a.add(q[1] + q[8] - q[0] - q[9], 1);
    }
    const i64 n = a.shift<ORDER == 4 ? 12 : 11>();  // 2^12 / 2880 = 1 + 1216/2880, 2^11 / 1680 = 1 + 368/1680
    const double f = to_double(n + mulhi(n, ORDER == 4 ? ratio(1216, 2880) : ratio(368, 1680)), e);
    return e <= kExpMax ? f : of_bits(0x7ff8000000000000ull);
}

// 60 Phi' of Eq. six at a cell from the split values of cells j-3 .. j+3 (the
// centre is not used): 45 A1 - 9 A2 + A3 in units of 2^8.
GBR_HD double grad60(const i64 (&m)[7], const int (&ex)[7])
{
    int e = kExpMin;
#pragma unroll
    for (int k = 0; k < 7; ++k) e = k != 3 && ex[k] > e ? ex[k] : e;
    i64 q[7];
#pragma unroll
    for (int k = 0; k < 7; ++k) q[k] = aligned(m[k], ex[k], e);
    Acc a;
    a.add(q[4] - q[2], 45);
    a.add(q[1] - q[5], 9);
    a.add(q[6] - q[0], 1);
    const double g = to_double(a.shift<8>(), e + 8);
    return e <= kExpMax ? g : of_bits(0x7ff8000000000000ull);
}

}  // namespace fx
}  // namespace gbr
