// Checks the bitwise FP64 / FP32 conversions (common.h: to_float, split, join, mul_pow2) against the
// plain ones, bit for bit: random mantissas at every exponent, ties and carries of the
// rounding, zeros, infinities and NaN.  Prints the number of cases that differ (a zero
// trailing part may have either sign).
#include "../paper_2004_09389_gb300/csrc/common.h"

#include <cstdio>
#include <limits>
#include <random>

using namespace hdg;

static bool same(float a, float b) { return bits_of(a) == bits_of(b) || (a != a && b != b); }
static bool same(double a, double b) { return bits_of(a) == bits_of(b) || (a != a && b != b); }

int main() {
    std::mt19937_64 gen(1);
    long wrong = 0;
    auto check = [&](double a) {
        const float hi = float(a), lo = float(a - double(hi));
        const float2 v = split(a);
        if (!same(to_float(a), hi) || !same(v.x, hi) || !(same(v.y, lo) || (v.y == 0.f && lo == 0.f))) ++wrong;
        if (!same(join(make_float2(hi, lo)), double(hi) + double(lo))) ++wrong;
        for (double p2 : {0x1p-1000, 0x1p-30, 1.0, 0x1p60, 0x1p900})
            if (!same(mul_pow2(a, p2), a * p2)) ++wrong;
    };
    const uint64_t low[] = {0, 1, 0x0fffffff, 0x10000000, 0x10000001, 0x1fffffff, 0x20000000, 0x2fffffff, 0x30000000,
                            0xfffffffffffffull, 0xfffffe0000000ull, 0xffffff0000000ull, 0xfffffefffffffull};
    for (uint64_t ex = 0; ex < 2048; ++ex)
        for (int s = 0; s < 2; ++s) {
            auto make = [&](uint64_t m) {
                const uint64_t u = uint64_t(s) << 63 | ex << 52 | (m & 0xfffffffffffffull);
                return double_of(uint32_t(u >> 32), uint32_t(u));
            };
            for (uint64_t m : low) check(make(m));
            for (int k = 0; k < 400; ++k) {
                const uint64_t m = gen();
                check(make(m));
                check(make(m & ~0x1fffffffull));                       // a float
                check(make((m & ~0x1fffffffull) | 0x10000000));        // halfway between two
            }
        }
    // pairs that are no split of a double: any exponent distance and sign
    for (int k = 0; k < 4000000; ++k) {
        const uint64_t r = gen();
        const float x = float_of(uint32_t(r)), scale = std::ldexp(1.f, -int((r >> 32) % 64));
        const float y = x * scale * float_of(0x3f800000u | uint32_t(gen() & 0x7fffff)) * ((r >> 40) & 1 ? 1.f : -1.f);
        if (!same(join(make_float2(x, y)), double(x) + double(y))) ++wrong;
    }
    const float inf = std::numeric_limits<float>::infinity(), nan = std::numeric_limits<float>::quiet_NaN();
    for (float x : {0.f, -0.f, 1.f, -1.f, 1.5f, inf, -inf, nan})
        for (float y : {0.f, -0.f, 1e-9f, -1e-9f, inf, nan})
            if (!same(join(make_float2(x, y)), double(x) + double(y))) ++wrong;
    std::printf("%ld\n", wrong);
    return 0;
}
