// Reciprocal and reciprocal square root of an FP64 value on the integer pipe.
//
// A division or rsqrt spends six to eight FP64 instructions (GB300: 111 clocks
// per warp and SM for rsqrt, 159 for a division, with the FP64 pipe the bound
// of the FP64 stage); the same Newton correction on 64-bit integers takes
// about 25 clocks of the otherwise idle integer pipe. From a 24-bit seed y0
// (the FP32 approximation instruction) the residual e, |e| < 2^-21, is formed
// exactly to 2^-62, and the series of the correction is summed in fixed point:
//   1/M       = y0 (1 + e + e^2 + ...),          e = 1 - M y0,
//   1/sqrt(M) = y0 (1 + e/2 + 3/8 e^2 + ...),    e = 1 - M y0^2
// (Newton and Halley, one step; the dropped terms are below 2^-62). Results
// are rounded to nearest from 62 bits: at most 0.51 ulp from the exact value.
// Zeros and subnormals give an infinity, infinities zero, NaN (and the rsqrt
// of a negative value) NaN; a reciprocal below the normal range gives zero.
// Below them: positive numbers as mantissa and exponent, for chains of products
// and roots, and a cell's primitives and fluxes on integers.
#pragma once

#include "fixed_face.cuh"

namespace gbr {
namespace fx {

GBR_HD float seed_bits(unsigned b)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    float f;
    memcpy(&f, &b, 4);
    return f;
#endif
}
GBR_HD unsigned float_bits(float f)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(f);
#else
    unsigned b;
    memcpy(&b, &f, 4);
    return b;
#endif
}
// y0 in (1/2, 1) as an integer of 24 bits (y0 2^24)
GBR_HD unsigned seed_mantissa(float y)
{
    const unsigned b = float_bits(y);
    return ((b < 0x3f7fffffu ? b : 0x3f7fffffu) & 0x7fffffu) | 0x800000u;
}
// y0 (1 + c) in units 2^-63, c in units 2^-63 (|c| < 2^43)
GBR_HD u64 corrected(unsigned y0, i64 c)
{
    const i64 t = ((i64)(int)(c >> 32) * (int)y0) * 256 + (i64)(((u64)(unsigned)c * y0) >> 24);
    return ((u64)y0 << 39) + (u64)t;
}

// 1 / M in units 2^-63, below 2^63, for M = m / 2^63 in [1, 2).
GBR_HD u64 rcp_mantissa(u64 m)
{
    const float f = seed_bits(0x3f800000u | ((unsigned)(m >> 40) & 0x7fffffu));
#ifdef __CUDA_ARCH__
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f));
#else
    const float y = 1.0f / f;
#endif
    const unsigned y0 = seed_mantissa(y);
    // e in units 2^-63: 2^63 - m y0 / 2^24
    const u64 p = (((u64)(unsigned)(m >> 32) * y0) << 8) + (((u64)(unsigned)m * y0) >> 24);
    const i64 r = (i64)(0x8000000000000000ull - p);
    const int h = (int)(r >> 21);
    const u64 R = corrected(y0, r + (((i64)h * h) >> 21));
    return R < 0x7fffffffffffffffull ? R : 0x7fffffffffffffffull;
}
// 1 / sqrt(M) in units 2^-63, below 2^63, for M = m / 2^63 in [1, 2), or twice that with `odd` = 1.
GBR_HD u64 rsqrt_mantissa(u64 m, int odd)
{
    const u64 X = m >> (1 - odd);  // M = X / 2^62
    const float f = seed_bits(0x3f800000u + ((unsigned)odd << 23) + ((unsigned)(m >> 40) & 0x7fffffu));
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f));
#else
    const float y = 1.0f / sqrtf(f);
#endif
    const unsigned y0 = seed_mantissa(y);
    // e in units 2^-62: 2^62 - X y0^2 / 2^48
    const i64 r = (i64)(0x4000000000000000ull - mulhi_u(X, ((u64)y0 * y0) << 16));
    const int h = (int)(r >> 20);
    const u64 R = corrected(y0, r + ((3 * ((i64)h * h)) >> 24));  // e/2 + 3/8 e^2 in units 2^-63
    return R < 0x7fffffffffffffffull ? R : 0x7fffffffffffffffull;
}

GBR_HD double rcp(double x)
{
    const u64 b = bits_of(x);
    const int e = (int)(b >> 52) & 0x7ff;
    const u64 R = rcp_mantissa((b << 11) | 0x8000000000000000ull);
    const u64 n = ((u64)(unsigned)(2044 - e) << 52) + (R >> 10) + ((R >> 9) & 1u);
    u64 s = e == 0 ? 0x7ff0000000000000ull : 0ull;
    s = (unsigned)(e - 1) < 2043u ? n : s;
    s = (b << 1) > 0xffe0000000000000ull ? 0x7ff8000000000000ull : s;  // NaN
    return of_bits(s | (b & 0x8000000000000000ull));
}

GBR_HD double rsqrt(double x)
{
    const u64 b = bits_of(x);
    const int e = (int)(b >> 52);  // (with the sign: a negative x is refused below)
    const int odd = (e + 1) & 1;   // exponent e - 1023 odd
    const u64 R = rsqrt_mantissa((b << 11) | 0x8000000000000000ull, odd);
    // x = M 2^(e - 1023 - odd): the result's biased exponent is that of 1/2 less half of it
    const u64 n = ((u64)(unsigned)(1021 - ((e - 1023 - odd) >> 1)) << 52) + (R >> 10) + ((R >> 9) & 1u);
    u64 s = (e & 0x7ff) == 0 ? 0x7ff0000000000000ull : 0x7ff8000000000000ull;
    s = b == 0x7ff0000000000000ull ? 0ull : s;
    return of_bits((unsigned)(e - 1) < 2046u ? n : s);
}

// Positive numbers (fixed_face.cuh): products are rounded down in the last of
// 63 bits.
GBR_HD Pos pos(u64 m, int e)  // m 2^(e - kOne), m > 0
{
    unsigned h = (unsigned)(m >> 32);
#ifdef __CUDA_ARCH__
    int n = h ? __clz((int)h) : 32 + __clz((int)(unsigned)m);
#else
    const int n = m ? __builtin_clzll(m) : 64;
#endif
    Pos r;
    r.m = m << (n & 63);
    r.e = e + 64 - kBits - n;
    return r;
}
GBR_HD Pos pos(double x)  // x positive and normal
{
    const u64 b = bits_of(x);
    Pos r;
    r.m = (b << 11) | 0x8000000000000000ull;
    r.e = (int)(b >> 52);
    return r;
}
GBR_HD Pos operator*(const Pos& a, const Pos& b)
{
    const u64 h = mulhi_u(a.m, b.m);  // M N / 2 in units 2^-63
    const int t = (int)(h >> 63);
    Pos r;
    r.m = t ? h : h << 1;
    r.e = a.e + b.e - 1023 + t;
    return r;
}
GBR_HD Pos rsqrt(const Pos& x)
{
    const int odd = (x.e + 1) & 1;
    Pos r;
    r.m = rsqrt_mantissa(x.m, odd) << 1;  // (1/2, 1) in units 2^-64
    r.e = 1022 - ((x.e - 1023 - odd) >> 1);
    return r;
}
GBR_HD Pos rcp(const Pos& x)
{
    Pos r;
    r.m = rcp_mantissa(x.m) << 1;
    r.e = 2045 - x.e;
    return r;
}
GBR_HD double to_double(const Pos& x)  // 1 <= e <= 2045
{
    return of_bits(((u64)(unsigned)(x.e - 1) << 52) + (x.m >> 11) + ((x.m >> 10) & 1u));
}

// The primitives and cell fluxes of one conservative cell (rho, rho u, rho v,
// E) on the integer pipe, as split values (integer of at most kBits bits, not
// necessarily normalised, and biased exponent): u = rho u / rho, v likewise, p
// = (gamma - 1) (E - (rho u u + rho v v) / 2). An FP64 evaluation rounds every
// step at 53 bits; here the steps keep 55 or more of their largest term. A density that is not
// positive and normal, or a value that is not finite, gives exponents that every
// later stencil refuses.
struct Split {
    i64 m;
    int e;
};
GBR_HD Split split(double x)
{
    Split r;
    unsigned short e;
    split(x, r.m, e);
    r.e = e;
    return r;
}
GBR_HD u64 magnitude(i64 x)
{
    const i64 g = x >> 63;
    return (u64)((x ^ g) - g);
}
GBR_HD Split product(const Split& a, const Split& b)
{
    const i64 g = (a.m ^ b.m) >> 63;
    Split r;
    r.m = ((i64)mulhi_u(magnitude(a.m) << (64 - kBits), magnitude(b.m)) ^ g) - g;
    r.e = a.e + b.e - 1022;
    return r;
}
GBR_HD Split sum(const Split& a, const Split& b)
{
    Split r;
    r.e = (a.e > b.e ? a.e : b.e) + 1;
    r.m = aligned(a.m, a.e, r.e) + aligned(b.m, b.e, r.e);
    return r;
}
// what the shared-memory planes hold: exponents in [1, 2047]
GBR_HD void store(const Split& x, i64& m, unsigned short& e)
{
    const int c = x.e < 1 ? 1 : x.e;
    m = x.e < 1 ? 0 : x.m;
    e = (unsigned short)(c > 2047 ? 2047 : c);
}
struct Cell {
    Split r, u, v, p, h;  // h = E + p
    Split ru, rv;         // rho u, rho v
    Split ruu, rvv;       // rho u u, rho v v
};
GBR_HD void cell_of(double q0, double q1, double q2, double q3, const Pos& gm1, Cell& c)
{
    c.r = split(q0);
    c.ru = split(q1);
    c.rv = split(q2);
    const Split E = split(q3);
    const u64 y = rcp_mantissa((u64)c.r.m << (64 - kBits));  // half of 2^1023 / rho in units of 2^(-64 - e)
    const bool bad = c.r.m <= 0 || larger(larger(c.r.e, c.ru.e), larger(c.rv.e, E.e)) == 2047;
    const int er = bad ? -4096 : 1023 - c.r.e;
    c.u.m = mulhi(c.ru.m, y) << 1;  // (the products below keep what their factors' leading bits leave)
    c.u.e = c.ru.e + er;
    c.v.m = mulhi(c.rv.m, y) << 1;
    c.v.e = c.rv.e + er;
    c.ruu = product(c.ru, c.u);
    c.rvv = product(c.rv, c.v);
    Split t;  // E - (rho u u + rho v v) / 2
    t.e = larger(E.e, larger(c.ruu.e, c.rvv.e) - 1) + 1;
    t.m = aligned(E.m, E.e, t.e) - aligned(c.ruu.m, c.ruu.e - 1, t.e) - aligned(c.rvv.m, c.rvv.e - 1, t.e);
    c.p.m = mulhi(t.m, gm1.m >> 1);
    c.p.e = t.e + gm1.e - 1021;
    if (bad) c.r.e = c.u.e = c.v.e = c.p.e = 2047;
    c.h = sum(E, c.p);
}

}  // namespace fx
}  // namespace gbr
