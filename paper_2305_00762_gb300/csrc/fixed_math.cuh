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

GBR_HD double rcp(double x)
{
    const u64 b = bits_of(x);
    const int e = (int)(b >> 52) & 0x7ff;
    const u64 m = (b << 11) | 0x8000000000000000ull;  // mantissa M = m / 2^63 in [1, 2)
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
    const int odd = (e + 1) & 1;   // exponent e - 1023 odd: M in [2, 4), else [1, 2)
    const u64 m = (b << 11) | 0x8000000000000000ull;
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
    // x = M 2^(e - 1023 - odd): the result's biased exponent is that of 1/2 less half of it
    const u64 n = ((u64)(unsigned)(1021 - ((e - 1023 - odd) >> 1)) << 52) + (R >> 10) + ((R >> 9) & 1u);
    u64 s = (e & 0x7ff) == 0 ? 0x7ff0000000000000ull : 0x7ff8000000000000ull;
    s = b == 0x7ff0000000000000ull ? 0ull : s;
    return of_bits((unsigned)(e - 1) < 2046u ? n : s);
}

}  // namespace fx
}  // namespace gbr
