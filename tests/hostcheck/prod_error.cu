// Host check of prod_error (dd_arith.cuh): on factor pairs over the whole
// binary64 range (products near the subnormals and the overflow threshold,
// subnormal factors, short significands, powers of two, zeros) it is the fused
// multiply-add's error, as a number.  Prints "pairs N bad M".
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>

#include "dd_arith.cuh"

static uint64_t state = 0x9E3779B97F4A7C15ull;
static uint64_t rnd() {
    state ^= state << 13;
    state ^= state >> 7;
    state ^= state << 17;
    return state * 0x2545F4914F6CDD1Dull;
}
static double pattern(int field) {
    static const uint64_t mants[8] = {0, 1, 0x8000000000000ull, 0xFFFFFFFFFFFFFull, 0xFFFFFFFFFFFFEull,
                                      0x7FFFFFFFFFFFFull, 0x100000000ull, 0xFFFFFFFFull};
    uint64_t m = (rnd() & 1) ? mants[rnd() % 8] : (rnd() & 0xFFFFFFFFFFFFFull);
    if (rnd() % 8 == 0) m >>= rnd() % 52;
    const uint64_t u = ((rnd() & 1) << 63) | ((uint64_t)field << 52) | m;
    double x;
    memcpy(&x, &u, 8);
    return x;
}

int main() {
    long pairs = 0, bad = 0;
    for (int it = 0; it < 6000000; ++it) {
        int fa = (int)(rnd() % 2047), fb = 0;
        switch (rnd() % 4) {
            case 0: fb = (int)(rnd() % 2047); break;
            case 1: fb = 1022 + (int)(rnd() % 120) - fa; break;        // about the least normal
            case 2: fb = 1045 + (int)(rnd() % 60) - fa; break;
            default: fb = 3069 - fa - (int)(rnd() % 4); break;         // about the largest
        }
        if (rnd() % 64 == 0) fa = 0;
        fb = fb < 0 ? 0 : fb > 2046 ? 2046 : fb;
        const double a = pattern(fa), b = pattern(fb);
        volatile double p = a * b;
        const double got = mpdd::prod_error(a, b, p);
        ++pairs;
        if (std::isinf(p) ? !std::isnan(got) : !(got == std::fma(a, b, -p))) ++bad;
    }
    printf("pairs %ld bad %ld\n", pairs, bad);
    return 0;
}
