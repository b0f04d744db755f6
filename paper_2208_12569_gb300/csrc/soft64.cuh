// Correctly rounded double-precision multiply, divide and square root on the
// integer pipe.
//
// GB300 issues a double-precision warp instruction every 64 cycles per SM
// partition (1.06 TFLOP/s of FMAs against 71 in single precision, measured),
// while integer instructions issue every cycle. The same IEEE 754 results (round
// to nearest, ties to even) are formed here from 32 x 32 -> 64-bit integer
// products: a quotient in about 100 issue slots (fewer when the divisor is
// shared) and a square root in about 110, each of which holds the FP64 pipe
// for about ten instructions, 640 cycles, as hardware code. The FP64 tracer
// with these two, and with the hardware's: 21.5 and 33.0 ms for a map of 512x512
// seeds, 80.8 and 126 ms for 1024x1024; four updates of a 256x256x128 gradient
// grid 6.2 and 15.5 ms. The multiply, about 35 slots, is correct too but loses to
// the pipe's 64 cycles in the tracer (trace64.cuh) and is used by nothing.
//
// The integer paths take operands with biased exponents in [768, 1279], that
// is 2^-255 <= |x| < 2^257, whose results can neither overflow nor be
// subnormal, and a zero divided by such a divisor or under the root; anything
// else (subnormals, infinities, NaNs, huge and tiny values) goes to the hardware
// operation. Both give the same bits, so which one runs shows in no result. All
// of it compiles for the host as well, where a test compares it with the
// processor's own operations.
//
// Methods: schoolbook products of 32-bit digits; quotient digits from a
// truncated reciprocal with an exact remainder (long division in base 2^28,
// Knuth, The Art of Computer Programming 2, Sec. 4.3.1); square root digits
// from a truncated reciprocal root with an exact remainder. The first
// approximations are the single-precision reciprocal and reciprocal square
// root with one Newton step; they only have to be good to a few units of 2^-22,
// the remainders make the result exact.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

namespace fqsl {
namespace soft64 {

#define FQSL_HD __host__ __device__ __forceinline__

FQSL_HD uint64_t bits_of(double x)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t b;
    memcpy(&b, &x, sizeof b);
    return b;
#endif
}

FQSL_HD double of_bits(uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double x;
    memcpy(&x, &b, sizeof x);
    return x;
#endif
}

FQSL_HD double of_words(uint32_t hi, uint32_t lo) { return of_bits(((uint64_t)hi << 32) | lo); }

FQSL_HD uint32_t float_bits(float x)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(x);
#else
    uint32_t b;
    memcpy(&b, &x, sizeof b);
    return b;
#endif
}

FQSL_HD float float_of(uint32_t b)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    float x;
    memcpy(&x, &b, sizeof x);
    return x;
#endif
}

FQSL_HD uint32_t mulhi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }

// 1/x and 1/sqrt(x) of a float, to a few units in the last place (the host
// stand-ins add an error of their own so that a test covers what a device's
// approximation may return)
FQSL_HD float rcp_approx(float x)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
#else
    return float_of(float_bits(1.0f / x) + (float_bits(x) % 5u) - 2u);
#endif
}

FQSL_HD float rsqrt_approx(float x)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
#else
    return float_of(float_bits(1.0f / sqrtf(x)) + (float_bits(x) % 5u) - 2u);
#endif
}

constexpr uint32_t kExpMask = 0x7ff00000u;
constexpr uint32_t kExpLow = 768u << 20;  // smallest exponent field of the integer paths

// 0 where the exponent field e (in place) is in range, else one of the top 3 bits set
FQSL_HD uint32_t out_of_range(uint32_t e) { return (e - kExpLow) & 0xe0000000u; }

// Operands outside the integer paths' range: the hardware operations, but for
// exact zeros over a divisor in range and under the root. Those are ordinary (a
// component of a field along an axis, J of a current-free one, the error of a
// straight line's step), and sent to the hardware they made a lane of each group
// wait for the FP64 pipe beside the others' integer quotients: FP64 map of 512x512
// seeds in a constant field of an anisotropic 128x128x64 cube 38.0 ms, 20.8 with
// this; gradient grid of a vertical field 256x128x64 2.0 ms, 0.55. (Out of line: the
// test in every quotient cost the gradient grid 3 %.)
#ifdef __CUDA_ARCH__
#define FQSL_OUTSIDE static __device__ __noinline__
static __device__ __forceinline__ double hw_div(double a, double b) { return __ddiv_rn(a, b); }
static __device__ __forceinline__ double hw_sqrt(double a) { return __dsqrt_rn(a); }
static __device__ __forceinline__ double hw_mul(double a, double b) { return __dmul_rn(a, b); }
#else
#define FQSL_OUTSIDE static inline
static inline double hw_div(double a, double b) { return a / b; }
static inline double hw_sqrt(double a) { return sqrt(a); }
static inline double hw_mul(double a, double b) { return a * b; }
#endif

FQSL_OUTSIDE double div_outside(double a, double b)
{
    const uint32_t ah = (uint32_t)(bits_of(a) >> 32), bh = (uint32_t)(bits_of(b) >> 32);
    if (!(bits_of(a) << 1) && !out_of_range(bh & kExpMask)) return of_words((ah ^ bh) & 0x80000000u, 0u);
    return hw_div(a, b);
}

FQSL_OUTSIDE double sqrt_outside(double x) { return bits_of(x) << 1 ? hw_sqrt(x) : x; }

// Round the 53-bit integer m (its leading bit set) with the fraction word r
// (units of 2^-32, its low bits sticky) to nearest, ties to even, and pack it
// with the exponent field e - 1 in place (the leading bit adds 1; a carry out of
// the mantissa moves the exponent up by itself) and the sign bit.
FQSL_HD double round_pack(uint64_t m, uint32_t r, uint32_t e_less_1, uint32_t sign)
{
    m += ((uint64_t)r + (0x7fffffffu + ((uint32_t)m & 1u))) >> 32;
    m += (uint64_t)e_less_1 << 32;
    return of_words((uint32_t)(m >> 32) | sign, (uint32_t)m);
}

// a factor ready for several products
struct Factor {
    double x;
    uint32_t m1, m0;  // mantissa << 11: 64 bits, the top one set
    uint32_t e, s;    // exponent field less 1023, in place; sign bit
    uint32_t bad;     // nonzero: outside the integer path's range
};

FQSL_HD Factor factor(double x)
{
    const uint64_t b = bits_of(x);
    const uint32_t h = (uint32_t)(b >> 32), l = (uint32_t)b;
    Factor f;
    f.x = x;
    f.m1 = (h << 11) | (l >> 21) | 0x80000000u;
    f.m0 = l << 11;
    f.s = h & 0x80000000u;
    f.e = (h & kExpMask) - (1023u << 20);
    f.bad = out_of_range(h & kExpMask);
    return f;
}

// x * f on the integer pipe, both in range
FQSL_HD double mul_in_range(double x, const Factor &f)
{
    const uint64_t b = bits_of(x);
    const uint32_t h = (uint32_t)(b >> 32), l = (uint32_t)b;
    const uint32_t a1 = (h & 0xfffffu) | 0x100000u;
    // (a1:l) (21 + 32 bits) times (m1:m0): hi = its bits 64 up (52 or 53 of them)
    const uint64_t p = (uint64_t)l * f.m0;
    const uint64_t t = (uint64_t)l * f.m1 + (p >> 32);
    const uint64_t u = (uint64_t)a1 * f.m0 + (uint32_t)t;
    uint64_t hi = (uint64_t)a1 * f.m1 + ((t >> 32) + (u >> 32));
    uint32_t r = (uint32_t)u | ((uint32_t)p != 0u ? 1u : 0u);
    uint32_t e = (h & kExpMask) + f.e;
    if (!(hi >> 52)) {
        hi = (hi << 1) | (r >> 31);
        r <<= 1;
        e -= 1u << 20;
    }
    return round_pack(hi, r, e, (h & 0x80000000u) ^ f.s);
}

FQSL_HD double mul64(double a, double b)
{
    const Factor f = factor(b);
    if (f.bad | out_of_range((uint32_t)(bits_of(a) >> 32) & kExpMask)) return hw_mul(a, b);
    return mul_in_range(a, f);
}

// a divisor ready for several quotients
struct Divisor {
    double x;
    uint64_t m;     // 53-bit mantissa
    uint32_t r;     // 2^31 / (m / 2^52), less at most 4
    uint32_t e, s;  // exponent field in place, sign bit
    uint32_t bad;
};

FQSL_HD Divisor divisor(double x)
{
    const uint64_t b = bits_of(x);
    const uint32_t h = (uint32_t)(b >> 32);
    Divisor d;
    d.x = x;
    d.m = (b & 0xfffffffffffffull) | (1ull << 52);
    d.e = h & kExpMask;
    d.s = h & 0x80000000u;
    d.bad = out_of_range(d.e);
    const uint32_t top = (uint32_t)(d.m >> 21);  // m / 2^52 = top / 2^31 (truncated)
    // a float above it, by more than the approximation's error, so that y is
    // below the reciprocal; y < 1
    const float y = rcp_approx(float_of(0x3f800008u + (top << 1 >> 9)));
    const uint32_t yb = float_bits(y);
    const uint32_t r0 = ((yb & 0x7fffffu) | 0x800000u) << (7 + (int)(yb >> 23) - 126);
    // y 2^31, and one Newton step: r0 top = 2^62 (1 - eps) with 0 < eps < 2^-19.
    // The truncated m lifts the result by one unit at most.
    const uint64_t e = (1ull << 62) - (uint64_t)r0 * top;
    d.r = r0 + (mulhi(r0, (uint32_t)(e >> 12)) >> 18) - 2u;
    return d;
}

// x / d on the integer pipe, both in range
FQSL_HD double div_in_range(double x, const Divisor &d)
{
    const uint64_t b = bits_of(x);
    const uint32_t h = (uint32_t)(b >> 32);
    uint64_t a = (b & 0xfffffffffffffull) | (1ull << 52);
    uint32_t e = (h & kExpMask) - d.e + (1022u << 20);
    if (a < d.m) {
        a <<= 1;
        e -= 1u << 20;
    }
    // a / m in [1, 2). Two digits, each less than 6 below the quotient that it
    // stands for (the reciprocal's 4, the truncated factor, the floor): q1 of
    // a 2^29 / m, q2 of rem1 2^27 / m.
    const uint32_t q1 = mulhi((uint32_t)(a >> 22), d.r);
    const uint64_t rem1 = (a << 29) - (uint64_t)q1 * d.m;  // < 6 m < 2^56
    const uint32_t q2 = mulhi((uint32_t)(rem1 >> 24), d.r);
    uint64_t rem = (rem1 << 27) - (uint64_t)q2 * d.m;
    uint64_t q = ((uint64_t)q1 << 27) + q2;  // a 2^56 / m = q + rem / m, rem < 6 m
    if (rem >= 4 * d.m) {
        rem -= 4 * d.m;
        q += 4;
    }
    if (rem >= 2 * d.m) {
        rem -= 2 * d.m;
        q += 2;
    }
    if (rem >= d.m) {
        rem -= d.m;
        q += 1;
    }
    const uint32_t r = ((uint32_t)q << 28) | (rem != 0 ? 1u : 0u);  // the 4 bits below the mantissa
    return round_pack(q >> 4, r, e, (h & 0x80000000u) ^ d.s);
}

FQSL_HD double div64(double a, const Divisor &d)
{
    if (d.bad | out_of_range((uint32_t)(bits_of(a) >> 32) & kExpMask)) return div_outside(a, d.x);
    return div_in_range(a, d);
}

FQSL_HD double div64(double a, double b) { return div64(a, divisor(b)); }

FQSL_HD double sqrt64(double x)
{
    const uint64_t b = bits_of(x);
    const uint32_t h = (uint32_t)(b >> 32);
    if (out_of_range(h)) return sqrt_outside(x);  // (a set sign bit is out of range too)
    // x = m 2^(2k - 52) with m / 2^52 in [1, 4)
    const uint32_t odd = ((h >> 20) & 1u) ^ 1u;  // (exponent less 1023) odd
    const uint64_t m = ((b & 0xfffffffffffffull) | (1ull << 52)) << odd;
    const uint32_t top = (uint32_t)(m >> 22);  // m / 2^52 = top / 2^30
    // y < 1 / sqrt(m / 2^52), from a float above m / 2^52 by more than the
    // approximation's error
    const float f = float_of((odd ? 0x40000010u : 0x3f800010u) + (uint32_t)((b >> 29) & 0x7fffffu));
    const uint32_t yb = float_bits(rsqrt_approx(f));
    const uint32_t y0 = ((yb & 0x7fffffu) | 0x800000u) << (7 + (int)(yb >> 23) - 126);  // y 2^31
    // one Newton step, y += y eps / 2 with eps = 1 - (m / 2^52) y^2 in (0, 2^-18)
    const uint32_t yy = mulhi(y0 << 1, y0 << 1);            // y^2 2^32
    const uint64_t ee = (1ull << 62) - (uint64_t)yy * top;  // eps 2^62
    const uint32_t y = y0 + (mulhi(y0, (uint32_t)(ee >> 12)) >> 19) - 3u;
    // first digit: sqrt(m / 2^52) 2^30, less than 16 below it
    const uint32_t s1 = mulhi(top, y) << 1;
    const uint64_t rem1 = (m << 8) - (uint64_t)s1 * s1;  // < 2^37
    // second digit: rem1 / (2 root) 2^26, less than 10 below it
    const uint32_t s2 = (uint32_t)(((uint64_t)(uint32_t)(rem1 >> 5) * y) >> 31);
    // s of sqrt(m / 2^52) 2^56; its remainder m 2^60 - s^2 fits 64 bits
    uint64_t s = ((uint64_t)s1 << 26) + s2;
    uint64_t rem = (m << 60) - s * s;
#pragma unroll
    for (int j = 8; j >= 1; j >>= 1) {
        // (s + j)^2 <= m 2^60
        const uint64_t c = 2 * (uint64_t)j * s + (uint64_t)(j * j);
        if (rem >= c) {
            rem -= c;
            s += (uint64_t)j;
        }
    }
    const uint32_t r = ((uint32_t)s << 28) | (rem != 0 ? 1u : 0u);  // the 4 bits below the mantissa
    return round_pack(s >> 4, r, ((((h >> 20) + 1023u) >> 1) - 1u) << 20, 0u);
}

}  // namespace soft64
}  // namespace fqsl
