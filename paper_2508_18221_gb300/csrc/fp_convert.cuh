// FP64 <-> FP32 conversions with integer instructions and selects, for the FP32 algebra of
// the mixed-precision modes; FP64 reciprocals (at the end).
//
// GB300 executes the hardware conversions (F2F) on its FP64 pipe, which issues about 1/64
// of the integer rate; kernels that convert every input and output (the FP32 right-hand
// side, the FP32 fluxes, the tensor-core line tiles) were bound by it.  Narrowing keeps the
// leading 23 bits of the FP64 mantissa, rounded to nearest even on the 29 dropped bits (a
// carry steps the exponent, up to Inf); widening appends 29 zero bits.  Both give the
// hardware's bits except below FP32's normal range (|x| < 2^-126 ~ 1.2e-38), which becomes
// a signed zero instead of an FP32 subnormal -- irrelevant at FP32 precision and keeping
// the code free of branches, which would stop the compiler from batching the loads that
// feed the conversions.  Inf and NaN stay Inf and NaN.
//
// The narrowing works on the whole word (exponent and mantissa shifted together, one addition
// that carries on a round-up) instead of on the fields: same bits, checked on the host on 2e8
// values, about a third fewer instructions; the FP32 right-hand side of 4,194,304 nodes, which
// converts some 60 values per node, went from 989 to 943 us.
#pragma once

#include <stdint.h>

namespace gk {

__device__ __forceinline__ float d2f_rn(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b, mag = hi & 0x7FFFFFFFu;
    const uint32_t a = mag - 0x38000000u;                        // exponent bias 1023 -> 127
    const uint32_t m = (a << 3) | (lo >> 29);                    // exponent and leading 23 mantissa bits
    // the dropped bits, at the top of a word, plus the last kept bit: above one half, or a tie to odd
    const uint32_t normal = m + ((lo << 3) + (m & 1u) > 0x80000000u ? 1u : 0u);
    const uint32_t big = mag > 0x7FF00000u || (mag == 0x7FF00000u && lo != 0u) ? 0x7FC00000u : 0x7F800000u;
    const uint32_t odd = (int)a < 0x00100000 ? 0u : big;         // below or above the normal range
    return __uint_as_float((a - 0x00100000u < 0x0FE00000u ? normal : odd) | (hi & 0x80000000u));
}

__device__ __forceinline__ double f2d(float f) {
    const uint32_t u = __float_as_uint(f);
    const uint32_t s = u & 0x80000000u, ef = (u >> 23) & 0xFFu, m = u & 0x7FFFFFu;
    const uint32_t eh = ef == 255u ? 0x7FF00000u : ((ef + 896u) << 20);
    return __hiloint2double((int)(ef == 0u ? s : (s | eh | (m >> 3))), (int)(ef == 0u ? 0u : (m << 29)));
}

// FP64 -> the mixed modes' algebra type, and back
template <class R> __device__ __forceinline__ R narrow(double x);
template <> __device__ __forceinline__ float narrow<float>(double x) { return d2f_rn(x); }
__device__ __forceinline__ double widen(float x) { return f2d(x); }

// Reciprocal and reciprocal square root: the hardware's 20-bit seeds (rcp / rsqrt.approx.f64)
// with one Householder step of third order, y (1 + e + e^2), e = 1 - x y, and
// y (1 + e/2 + 3 e^2 / 8), e = 1 - x y^2, in 3 and 5 FP64 instructions (1.0 / x and rsqrt(x) take
// about twice as many, and the FP64 pipe bounds the kernels here).  Over 4e6 values of every
// exponent both are within 0.507 units in the last place (rsqrt(x) too; 1 value in 460 of the
// reciprocals differs from 1.0 / x).  Operands near the ends of the exponent range, zero, Inf,
// NaN and negative ones take the library functions.
static __device__ __noinline__ double rcp64_any(double x) { return 1.0 / x; }
static __device__ __noinline__ double rsqrt64_any(double x) { return rsqrt(x); }
__device__ __forceinline__ double rcp64(double x) {
    const unsigned ex = ((unsigned)__double2hiint(x) >> 20) & 0x7FFu;
    if (ex - 64u > 1918u) return rcp64_any(x);
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ double rsqrt64(double x) {
    const unsigned ex = (unsigned)__double2hiint(x) >> 20;    // with the sign: negative is out of range
    if (ex - 64u > 1918u) return rsqrt64_any(x);
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y * y, 1.0);                      // y * y is exact: the seed's low word is zero
    return fma(y, e * fma(0.375, e, 0.5), y);
}

}  // namespace gk
