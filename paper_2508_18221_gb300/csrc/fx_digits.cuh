// Fixed-point digits of FP64 values and back, shared by the two digit-slice contractions
// (kernels_fx.cu on the tensor cores, kernels_fxs.cu on the integer units).
#pragma once

#include <stdint.h>

namespace gk {

constexpr unsigned long long DIG_BIAS = 0x80808080808080ull;  // 128 in each digit

// Digit word of one value: Z = X + bias with X = round(2 m 2^(e - EL)) the value as a
// signed fixed-point integer relative to the line exponent EL (|X| <= 2^54; the value is
// X 2^(EL - 1076)); byte b of Z minus 128 is the balanced digit of weight 256^b.  Branch-
// free (the values of a thread overlap): with y = +-(4 m >> sh), sh = EL - e in 0 .. 63
// (4 m < 2^56, so every sh >= 56 gives 0; zero for e = 0), X + bias is (y + 1 + 2 bias) >> 1
// for y >= 0 and (y + 2 bias) >> 1 = (~|y| + 1 + 2 bias) >> 1 below: sign, rounding (to the
// nearest, halves away from zero) and bias in one 64-bit addition to the magnitude or its
// complement.  The integer pipes bound the conversion, so the shift by two is left to the
// multiply-add pipe (four).
__device__ __forceinline__ unsigned long long digit_word(double u, int EL, uint32_t four) {
    const uint32_t hi = (uint32_t)__double2hiint(u), lo = (uint32_t)__double2loint(u);
    const int e = (int)((hi >> 20) & 0x7FFu);
    const unsigned long long m4 =
        (unsigned long long)lo * four + ((unsigned long long)(((hi & 0xFFFFFu) | 0x100000u) * four) << 32);
    const int sh = e != 0 ? min(EL - e, 63) : 63;
    const unsigned long long y = m4 >> sh;
    const uint32_t s = (uint32_t)((int)hi >> 31);
    const unsigned long long ys = y ^ (((unsigned long long)s << 32) | s);
    return (ys + (2 * DIG_BIAS + 1)) >> 1;
}

// R * 2^X: one correctly rounded integer-to-double conversion, then the power of two is
// added to the exponent field; *ok false when the result leaves the normal range or R = 0
// (the caller then takes ldexp_int below).  Branch-free, so that the eight outputs of a
// column block overlap their conversions.
__device__ __forceinline__ double ldexp_int(long long R, int X);
__device__ __forceinline__ double scale_int_fast(long long R, int X, bool* ok) {
    const double v = __ll2double_rn(R);
    const int lo = __double2loint(v), hi = __double2hiint(v);
    const int e = (hi >> 20) & 0x7FF;
    *ok = e != 0 && (unsigned)(e + X - 1) < 2046u;
    return __hiloint2double(hi + (X << 20), lo);
}

// R * 2^X as an IEEE double built with integer instructions (|R| < 2^62; ties away)
__device__ __forceinline__ double ldexp_int(long long R, int X) {
    if (R == 0) return 0.0;
    const unsigned long long sgn = R < 0 ? (1ull << 63) : 0ull;
    const unsigned long long a = R < 0 ? (unsigned long long)(-R) : (unsigned long long)R;
    const int p = 63 - __clzll((long long)a);
    unsigned long long mant;
    if (p <= 52) mant = a << (52 - p);
    else { const int sh = p - 52; mant = (a + (1ull << (sh - 1))) >> sh; }
    const int be = p + X + 1023;
    if (be <= 0) return __longlong_as_double((long long)sgn);
    if (be >= 2047) return __longlong_as_double((long long)(sgn | 0x7FF0000000000000ull));
    return __longlong_as_double((long long)(sgn | ((((unsigned long long)(be - 1)) << 52) + mant)));
}

}  // namespace gk
