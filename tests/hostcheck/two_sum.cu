// Host check of two_sum (dd_arith.cuh): on operand pairs over the whole
// binary64 range (equal and adjacent exponents, ties, powers of two,
// cancellation, subnormals, zeros) its s and e, and sum_error, are those of
// Knuth's six operations, as numbers, in either operand order.  Prints
// "pairs N bad M".
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>

#include "dd_arith.cuh"

static uint64_t state = 88172645463325252ull;
static uint64_t rnd() {
    state ^= state << 13;
    state ^= state >> 7;
    state ^= state << 17;
    return state;
}

static double pattern(int field) {
    static const uint64_t mants[8] = {0, 1, 0x8000000000000ull, 0xFFFFFFFFFFFFFull, 0xFFFFFFFFFFFFEull,
                                      0x7FFFFFFFFFFFFull, 0x100000000ull, 0xFFFFFFFFull};
    const uint64_t m = (rnd() & 1) ? mants[rnd() % 8] : (rnd() & 0xFFFFFFFFFFFFFull);
    const uint64_t u = ((rnd() & 1) << 63) | ((uint64_t)field << 52) | m;
    double x;
    memcpy(&x, &u, 8);
    return x;
}

int main() {
    long pairs = 0, bad = 0;
    for (int it = 0; it < 4000000; ++it) {
        const int f = (int)(rnd() % 2045);
        int d = (int)(rnd() % 5);
        d = d == 0 ? 0 : d == 1 ? 1 : d == 2 ? (int)(rnd() % 4) : d == 3 ? (int)(rnd() % 60) : (int)(rnd() % 2000);
        const double a = pattern(f);
        double b = pattern(f > d ? f - d : 0);
        if (it % 16 == 0) b = -a;
        if (it % 31 == 0) b = 0.0;
        for (int order = 0; order < 2; ++order) {
            const double x = order ? b : a, y = order ? a : b;
            volatile double s = x + y;
            volatile double bv = s - x, av = s - bv;
            volatile double ra = x - av, rb = y - bv, e = ra + rb;
            double s2, e2;
            mpdd::two_sum(x, y, s2, e2);
            ++pairs;
            if (std::isinf(s)) continue;   // (both error words are non-finite)
            if (!(s2 == s && e2 == e && mpdd::sum_error(x, y, s) == e)) ++bad;
        }
    }
    printf("pairs %ld bad %ld\n", pairs, bad);
    return 0;
}
