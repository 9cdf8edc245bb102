// BF16 planes of a double cut from two_floats (split.cuh): p planes of a value in [2^e, 2^(e+1)) leave at most half
// a unit of the last one, 2^-8, 2^-17 and 2^-26 times 2^e for one, two and three planes, where the remainders are
// exact.  Here a remainder's leading FP32 decides its rounding, which can move what it leaves by 2^-15 of itself;
// a rounding of x to FP32 before the cut leaves 2^-25 after three planes.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>

#include "split.cuh"

// nearest BF16, ties to even
static float bf16(float f) {
    uint32_t u;
    std::memcpy(&u, &f, 4);
    u = (u + 0x7fffu + ((u >> 16) & 1u)) & 0xffff0000u;
    std::memcpy(&f, &u, 4);
    return f;
}
static int bad = 0;
static double worst[3];

static void one(double x) {
    float hi, lo;
    adc::two_floats(x, hi, lo);
    if (!(std::fabs(x - ((double)hi + (double)lo)) <= std::ldexp(std::fabs(x), -46))) {
        if (bad++ < 5) std::printf("%a: hi + lo = %a + %a\n", x, hi, lo);
    }
    float f = adc::odd(hi, lo);
    double left = x;
    const double unit = std::ldexp(1.0, std::ilogb(x));
    for (int p = 0; p < 3; ++p) {
        const float h = bf16(f);
        f = adc::add_keep((p == 0 ? hi : f) - h, lo);
        left -= (double)h;
        if (!(std::fabs(left) <= std::ldexp(unit, -9 * p - 8) * (1 + 0x1p-14)) && bad++ < 5)
            std::printf("%a: %d planes leave %a\n", x, p + 1, left);
        worst[p] = std::fmax(worst[p], std::fabs(left) / unit);
    }
}

int main() {
    std::mt19937_64 g(1);
    std::uniform_real_distribution<double> u(-1.0, 1.0);
    for (int i = 0; i < 2000000; ++i) one(std::ldexp(u(g), (int)(g() % 160) - 80));
    // near the ties of the first and of the second plane, where a rounding to FP32 before the cut decides wrongly
    for (int i = 0; i < 2000000; ++i) {
        const double top = std::ldexp((double)(128 + g() % 128), -7), tie = std::ldexp((double)(2 * (g() % 128) + 1), -16);
        const double off = std::ldexp(u(g), -18 - (int)(g() % 30));
        const double x = i & 1 ? top + std::ldexp(1.0, -8) + off : top + tie + off;
        one(g() & 1 ? x : -x);
    }
    float hi, lo;
    for (double x : {0.0, -0.0, 1e-320, -4e-310}) {
        adc::two_floats(x, hi, lo);
        if (hi != 0.0f || lo != 0.0f || std::signbit(hi) != std::signbit(x)) ++bad, std::printf("%a\n", x);
    }
    for (double x : {(double)INFINITY, -(double)INFINITY, 1e300, -1e300}) {
        adc::two_floats(x, hi, lo);
        if (!std::isinf(hi) || lo != 0.0f) ++bad, std::printf("%a\n", x);
    }
    adc::two_floats(NAN, hi, lo);
    if (!std::isnan(hi)) ++bad;
    for (double x : {0x1.fffffffffffffp126, 0x1.fdp127, -0x1.8p-100, 0x1p-126, 0x1.fffffffffffffp-74, 0x1p-74}) one(x);
    std::printf("left after 1, 2, 3 planes: %a %a %a; %d wrong\n", worst[0], worst[1], worst[2], bad);
    return bad ? 1 : 0;
}
