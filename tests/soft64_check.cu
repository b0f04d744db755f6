// Host check of csrc/soft64.cuh against the processor's own double-precision
// multiply, divide and square root, bit for bit: random mantissas at every
// exponent distance, mantissas with long runs of zeros and ones (results at and
// beside ties and powers of two), exact products and squares, and the values
// outside the integer paths' range. Prints the number of results compared and
// of mismatches.
#include <stdio.h>
#include <stdlib.h>

#include "soft64.cuh"

using namespace fqsl::soft64;

static uint64_t state = 88172645463325252ull;
static uint64_t rnd()
{
    state ^= state << 13;
    state ^= state >> 7;
    state ^= state << 17;
    return state * 2685821657736338717ull;
}

static uint64_t mantissa()
{
    const uint64_t r = rnd();
    switch (r & 7u) {
    case 0: return (rnd() >> 12) & ~((1ull << (rnd() % 52u)) - 1u);  // trailing zeros
    case 1: return (rnd() >> 12) | ((1ull << (rnd() % 52u)) - 1u);   // trailing ones
    case 2: return (rnd() % 3u) == 0 ? 0u : ((1ull << 52) - 1u) >> (rnd() % 52u);
    case 3: return ((1ull << 52) - 1u) - (rnd() % 64u);
    case 4: return rnd() % 64u;
    case 5: return (rnd() & 0x7fffffull) << 29;  // a float's
    default: return rnd() >> 12;
    }
}

static double value(int lo, int hi)
{
    const uint64_t e = (uint64_t)(lo + (int)(rnd() % (uint64_t)(hi - lo + 1)));
    return of_bits((rnd() & 0x8000000000000000ull) | (e << 52) | mantissa());
}

static long long n = 0, bad = 0;
static void same(double got, double want, const char *what, double a, double b)
{
    n++;
    if (want != want ? got != got : bits_of(got) == bits_of(want)) return;
    if (bad++ < 10) printf("%s(%a, %a) = %a, not %a\n", what, a, b, got, want);
}

static void all(double a, double b)
{
    volatile double m = a * b, d = a / b;
    same(mul64(a, b), m, "mul", a, b);
    same(div64(a, b), d, "div", a, b);
    volatile double q = ::sqrt(a);
    same(sqrt64(a), q, "sqrt", a, 0.0);
}

int main(int argc, char **argv)
{
    const long long count = argc > 1 ? atoll(argv[1]) : 20000000;
    for (long long i = 0; i < count; i++) {
        const double a = value(768, 1279), b = value(768, 1279);
        all(a, b);
        if (i % 4 == 0) {  // quotients and roots that are exact, or one unit beside
            const double s = of_bits((1023ull << 52) | (rnd() >> 12 & ~((1ull << 27) - 1u)));
            const double t = of_bits((1023ull << 52) | (rnd() >> 12 & ~((1ull << 27) - 1u)));
            const uint64_t p = bits_of(s * t);
            for (int k = -1; k <= 1; k++) {
                all(of_bits(p + (uint64_t)(int64_t)k), t);
                all(of_bits(bits_of(s * s) + (uint64_t)(int64_t)k), s);
            }
        }
        if (i % 16 == 0) all(value(0, 2047), value(0, 2047));
    }
    const double edge[] = {0.0, -0.0, INFINITY, -INFINITY, NAN, 5e-324, -5e-324, 2.2250738585072014e-308,
                           1.7976931348623157e308, 0x1p-255, 0x1.fffffffffffffp-256, 0x1p256, 0x1.fffffffffffffp256,
                           0x1p257, 1.0, -1.0, 0x1.fffffffffffffp0, 0x1.0000000000001p0, 3.0};
    for (double a : edge)
        for (double b : edge) all(a, b);
    printf("%lld %lld\n", n, bad);
    return bad != 0;
}
