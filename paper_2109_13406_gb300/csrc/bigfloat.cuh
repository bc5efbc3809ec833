// Binary floating point with a 128-bit significand held in four 32-bit
// integer registers: the exact rounding of the residue (CRT) form's
// reconstructed integer to dd, and that of the digit form's recombined one
// (signed160_to_dd, which keeps all 160 bits).
//
// The reconstructed product Z 2^s is an exact multiword integer; its leading
// 128 bits are taken with integer instructions and rounded to the nearest dd
// (hi = RN(x), lo = RN(x - hi)).  On this GPU an FP64 operation issues at
// about 2 per clock per SM against 64 for integer ALU work, so the rounding
// stays off the FP64 pipe, which the alpha/beta epilogue uses.
//
// Accuracy: the bits below the leading 128 are dropped (relative error below
// 2^-127), so |x - (hi + lo)| <= (2^-106 + 2^-126) |x|.
#pragma once

#include <cstdint>
#include <cstring>

namespace mpdd {
namespace bigf {

#define BF_HD __host__ __device__ __forceinline__

// value = (-1)^neg * M * 2^(e - 127), M = m[3]:m[2]:m[1]:m[0] with bit 127
// set; M = 0 (m[3] == 0) is zero.
struct BF {
    uint32_t m[4];
    int e;
    uint32_t neg;
};

BF_HD int clz32(uint32_t x) {
#if defined(__CUDA_ARCH__)
    return __clz((int)x);
#else
    return x ? __builtin_clz(x) : 32;
#endif
}

BF_HD int clz64(uint64_t x) {
#if defined(__CUDA_ARCH__)
    return __clzll((long long)x);
#else
    return x ? __builtin_clzll(x) : 64;
#endif
}

// (hi:lo << s) >> 32 for 0 <= s <= 31.
BF_HD uint32_t fshl(uint32_t lo, uint32_t hi, int s) {
#if defined(__CUDA_ARCH__)
    return __funnelshift_l(lo, hi, s);
#else
    return (uint32_t)(((((uint64_t)hi << 32) | lo) << s) >> 32);
#endif
}
BF_HD double bitsd(uint64_t u) {
#if defined(__CUDA_ARCH__)
    return __longlong_as_double((long long)u);
#else
    double x;
    memcpy(&x, &u, 8);
    return x;
#endif
}

BF_HD BF bf_zero() {
    BF r;
    r.m[0] = r.m[1] = r.m[2] = r.m[3] = 0;
    r.e = 0;
    r.neg = 0;
    return r;
}

BF_HD bool is_zero(const BF &a) { return a.m[3] == 0; }

// M << s for 0 <= s < 128.
BF_HD void shl128(uint32_t (&m)[4], int s) {
    if (s <= 0) return;
    const int w = s >> 5, b = s & 31;
    const uint32_t t3 = w == 0 ? m[3] : w == 1 ? m[2] : w == 2 ? m[1] : m[0];
    const uint32_t t2 = w == 0 ? m[2] : w == 1 ? m[1] : w == 2 ? m[0] : 0u;
    const uint32_t t1 = w == 0 ? m[1] : w == 1 ? m[0] : 0u;
    const uint32_t t0 = w == 0 ? m[0] : 0u;
    m[3] = fshl(t2, t3, b);
    m[2] = fshl(t1, t2, b);
    m[1] = fshl(t0, t1, b);
    m[0] = t0 << b;
}

// Leading zeros of the 128-bit M (128 for zero).
BF_HD int clz128(const uint32_t (&m)[4]) {
    return m[3] ? clz32(m[3])
                : m[2] ? 32 + clz32(m[2]) : m[1] ? 64 + clz32(m[1]) : m[0] ? 96 + clz32(m[0]) : 128;
}

// |Z| 2^s for the magnitude words z (little endian), with sign neg.  The top
// 128 bits are kept (the bits below them truncated: relative error < 2^-127).
template <int NW>
BF_HD BF from_words(const uint32_t (&z)[NW], uint32_t neg, int s) {
    int p = -1;
#pragma unroll
    for (int t = 0; t < NW; ++t)
        if (z[t] != 0) p = t;
    BF r = bf_zero();
    if (p < 0) return r;
    uint32_t w4 = 0, w3 = 0, w2 = 0, w1 = 0, w0 = 0;
#pragma unroll
    for (int t = 0; t < NW; ++t) {
        if (p == t) {
            w4 = z[t];
            w3 = t >= 1 ? z[t - 1] : 0u;
            w2 = t >= 2 ? z[t - 2] : 0u;
            w1 = t >= 3 ? z[t - 3] : 0u;
            w0 = t >= 4 ? z[t - 4] : 0u;
        }
    }
    const int lz = clz32(w4);
    r.m[3] = fshl(w3, w4, lz);
    r.m[2] = fshl(w2, w3, lz);
    r.m[1] = fshl(w1, w2, lz);
    r.m[0] = fshl(w0, w1, lz);
    r.e = 32 * p + 31 - lz + s;
    r.neg = neg;
    return r;
}

// m 2^e (m < 2^53) as a binary64 with the sign bit sg; the exponent field
// is assembled directly when the result is normal, else (overflow or a
// subnormal result) the FP64 unit scales it.
BF_HD double make_double(uint64_t m, int e, uint32_t sg) {
    if (m == 0) return sg ? -0.0 : 0.0;
    const int top = 63 - clz64(m);
    const int E = top + e + 1023;
    if (top == 52 && E >= 1 && E <= 2046)
        return bitsd(((uint64_t)sg << 63) | ((uint64_t)E << 52) | (m & ((1ull << 52) - 1)));
    // rare: subnormal or overflowing result (m < 2^53 is exact in binary64)
    double x = (double)m;
    int k = e;
    while (k > 1000) {
        x *= 0x1p1000;
        k -= 1000;
    }
    while (k < -1000) {
        x *= 0x1p-1000;
        k += 1000;
    }
    x *= bitsd((uint64_t)(k + 1023) << 52);
    return sg ? -x : x;
}

// The nearest dd: hi = RN(x), lo = RN(x - hi) (ties to even), for the
// 128-bit significand (bits below it are treated as zero).
BF_HD void to_dd(const BF &x, double &hi, double &lo) {
    if (is_zero(x)) {
        hi = 0.0;
        lo = 0.0;
        return;
    }
    // hi: significand bits 127..75; round bit 74; the remainder R = bits 0..74
    uint64_t mh = ((uint64_t)x.m[3] << 21) | (x.m[2] >> 11);
    const uint32_t r2 = x.m[2] & 0x7FFu, r1 = x.m[1], r0 = x.m[0];
    const bool rbit = (r2 >> 10) & 1u;
    const bool sticky = (r2 & 0x3FFu) | r1 | r0;
    const bool up = rbit && (sticky || (mh & 1u));
    // |x - hi| in units of 2^(e - 127): R, or 2^75 - R when rounded up
    uint32_t l2 = r2, l1 = r1, l0 = r0;
    if (up) {
        uint64_t d = (uint64_t)0 - r0;
        l0 = (uint32_t)d;
        d = (uint64_t)0 - r1 - (d >> 63);
        l1 = (uint32_t)d;
        d = (uint64_t)0x800u - r2 - (d >> 63);
        l2 = (uint32_t)d;
        mh += 1;
    }
    hi = make_double(mh, x.e - 52, x.neg);   // mh <= 2^53: exact
    // lo = RN(L 2^(e - 127)), L < 2^75 in l2:l1:l0
    const uint32_t lsg = x.neg ^ (up ? 1u : 0u);
    uint32_t m[4] = {l0, l1, l2, 0u};
    const int lz = clz128(m);
    if (lz == 128) {
        lo = 0.0;
        return;
    }
    shl128(m, lz);                               // L's leading bit at 127
    uint64_t ml = ((uint64_t)m[3] << 21) | (m[2] >> 11);
    const bool lr = (m[2] >> 10) & 1u;
    const bool ls = (m[2] & 0x3FFu) | m[1] | m[0];
    if (lr && (ls || (ml & 1u))) ml += 1;
    // L's leading bit is bit (127 - lz) of the frame 2^(e - 127)
    lo = make_double(ml, x.e - 127 + (127 - lz) - 52, lsg);
}

// The nearest dd of Z 2^s for a two's complement Z of NW words (|Z| below
// 2^(32 NW - 1)): the same result, bit for bit, as from_words and to_dd on
// the magnitude.  The usual case (Z's leading bit in its upper two words, no
// carry of the negation into the leading words, a remainder with its leading
// bit among the first 32, exponents well inside the normal range) is written
// out: the five leading words are taken as they are or one word lower, the
// sign is an exclusive or, and both significands are assembled by adding the
// exponent field to the rounded bits.  About 75 integer instructions; the
// general path selects among all words and shifts by any count.
template <int NW>
BF_HD void signed_words_to_dd(const uint32_t (&S)[NW], int s, double &hi, double &lo) {
    const uint32_t mask = (S[NW - 1] >> 31) ? 0xFFFFFFFFu : 0u;
    const bool low = S[NW - 1] == mask;          // the top word is empty
    uint32_t below = 0;                          // the words under the leading five
#pragma unroll
    for (int t = 0; t + 6 < NW; ++t) below |= S[t];
    if (NW >= 6 && !low) below |= S[NW - 6];
    const uint32_t w4 = (low ? S[NW - 2] : S[NW - 1]) ^ mask;
    const uint32_t w3 = (low ? S[NW - 3] : S[NW - 2]) ^ mask;
    const uint32_t w2 = (low ? S[NW - 4] : S[NW - 3]) ^ mask;
    const uint32_t w1 = (low ? S[NW - 5] : S[NW - 4]) ^ mask;
    const uint32_t w0 = (low ? S[NW - 6] : S[NW - 5]) ^ mask;
    const int lz = clz32(w4);
    const int e = 32 * (NW - 1) + 31 - (low ? 32 : 0) - lz + s;
    const uint32_t m3 = fshl(w3, w4, lz), m2 = fshl(w2, w3, lz), m1 = fshl(w1, w2, lz),
                   m0 = fshl(w0, w1, lz);
    // hi: bits 127 .. 75, rounded by bit 74 and the rest
    const uint32_t r2 = m2 & 0x7FFu;
    const uint32_t ml = (m3 << 21) | (m2 >> 11);
    const bool up = (r2 >> 10) && (((r2 & 0x3FFu) | m1 | m0) != 0 || (ml & 1u));
    // lo: the remainder, or 2^75 minus it when rounded up
    const uint64_t r10 = ((uint64_t)m1 << 32) | m0;
    const uint64_t l10 = up ? 0 - r10 : r10;
    const uint32_t l2 = up ? 0x800u - r2 - (r10 != 0) : r2;
    const uint32_t l1 = (uint32_t)(l10 >> 32), l0 = (uint32_t)l10;
    const uint32_t a2 = (l2 << 21) | (l1 >> 11), a1 = (l1 << 21) | (l0 >> 11), a0 = l0 << 21;
    if (w4 == 0 || (mask != 0 && below == 0) || a2 == 0 || e < -900 || e > 1000) {
        uint32_t z[NW];                          // the magnitude
        uint32_t c = mask & 1u;
#pragma unroll
        for (int t = 0; t < NW; ++t) {
            const uint64_t v = (uint64_t)(S[t] ^ mask) + c;
            z[t] = (uint32_t)v;
            c = (uint32_t)(v >> 32);
        }
        to_dd(from_words<NW>(z, mask & 1u, s), hi, lo);
        return;
    }
    const uint64_t mh = ((uint64_t)(m3 >> 11) << 32) | ml;   // 2^52 <= mh < 2^53
    hi = bitsd((((uint64_t)(uint32_t)(e + 1022) << 52) + mh + (up ? 1 : 0)) |
               ((uint64_t)(mask & 1u) << 63));
    const int lz2 = clz32(a2);
    const uint32_t n2 = fshl(a1, a2, lz2), n1 = fshl(a0, a1, lz2), n0 = a0 << lz2;
    const uint32_t nl = (n2 << 21) | (n1 >> 11);
    const bool up2 = ((n1 >> 10) & 1u) && (((n1 & 0x3FFu) | n0) != 0 || (nl & 1u));
    const uint64_t nh = ((uint64_t)(n2 >> 11) << 32) | nl;
    lo = bitsd((((uint64_t)(uint32_t)(e - 53 - lz2 + 1022) << 52) + nh + (up2 ? 1 : 0)) |
               ((uint64_t)((mask & 1u) ^ (up ? 1u : 0u)) << 63));
}

// The nearest dd of V 2^s for a two's complement V of six words, |V| < 2^160:
// hi = RN(V 2^s), lo = RN(V 2^s - hi), every bit of V taking part (barring
// results near the ends of the exponent range).  The magnitude's five words
// are formed first, so both signs go the same way: 128 leading bits and a tail
// word of those below.  Written out is the usual case (V's leading bit in its
// fifth word, the remainder's among its first 32, exponents well inside the
// normal range); the general path covers the rest.
BF_HD void signed160_to_dd(const uint32_t (&S)[6], int s, double &hi, double &lo) {
    const uint32_t neg = S[5] >> 31, mask = 0u - neg;
    uint32_t z[5], c = neg;
#pragma unroll
    for (int t = 0; t < 5; ++t) {
        const uint64_t v = (uint64_t)(S[t] ^ mask) + c;
        z[t] = (uint32_t)v;
        c = (uint32_t)(v >> 32);
    }
    const int lz = clz32(z[4]);
    const int e = 159 - lz + s;
    const uint32_t m3 = fshl(z[3], z[4], lz), m2 = fshl(z[2], z[3], lz), m1 = fshl(z[1], z[2], lz),
                   m0 = fshl(z[0], z[1], lz), mt = fshl(0u, z[0], lz);
    // hi: the leading 53 bits, rounded by the next one and the rest
    const uint32_t r2 = m2 & 0x7FFu;
    const uint64_t r0 = ((uint64_t)m0 << 32) | mt;
    const bool rest = (m1 | m0 | mt) != 0;
    const uint32_t ml = (m3 << 21) | (m2 >> 11);
    const bool up = (r2 >> 10) && ((r2 & 0x3FFu) != 0 || rest || (ml & 1u));
    // lo: the remainder (107 bits), or 2^107 minus it when rounded up
    const uint64_t l0t = up ? 0 - r0 : r0;
    const uint32_t l0 = (uint32_t)(l0t >> 32), lt = (uint32_t)l0t;
    const uint32_t l1 = up ? 0u - m1 - (r0 != 0) : m1;
    const uint32_t l2 = up ? 0x800u - r2 - rest : r2;
    const uint32_t a2 = (l2 << 21) | (l1 >> 11), a1 = (l1 << 21) | (l0 >> 11),
                   a0 = (l0 << 21) | (lt >> 11), at = lt << 21;
    const uint32_t lneg = neg ^ (up ? 1u : 0u);
    if (z[4] == 0 || a2 == 0 || e < -900 || e > 1000) {
        if (z[4] == 0) {   // 128 bits: to_dd has them all
            const uint32_t w[4] = {z[0], z[1], z[2], z[3]};
            to_dd(from_words<4>(w, neg, s), hi, lo);
            return;
        }
        hi = make_double((((uint64_t)m3 << 21) | (m2 >> 11)) + (up ? 1 : 0), e - 52, neg);
        uint32_t m[4] = {lt, l0, l1, l2};
        const int lz2 = clz128(m);
        if (lz2 == 128) {
            lo = 0.0;
            return;
        }
        shl128(m, lz2);
        uint64_t mh = ((uint64_t)m[3] << 21) | (m[2] >> 11);
        if (((m[2] >> 10) & 1u) && (((m[2] & 0x3FFu) | m[1] | m[0]) != 0 || (mh & 1u))) mh += 1;
        // the remainder's leading bit is bit 127 - lz2 of the frame 2^(e - 159)
        lo = make_double(mh, e - 159 + (127 - lz2) - 52, lneg);
        return;
    }
    const uint64_t mh = ((uint64_t)(m3 >> 11) << 32) | ml;   // 2^52 <= mh < 2^53
    hi = bitsd((((uint64_t)(uint32_t)(e + 1022) << 52) + mh + (up ? 1 : 0)) |
               ((uint64_t)neg << 63));
    const int lz2 = clz32(a2);
    const uint32_t n2 = fshl(a1, a2, lz2), n1 = fshl(a0, a1, lz2), n0 = fshl(at, a0, lz2),
                   nt = fshl(0u, at, lz2);
    const uint32_t nl = (n2 << 21) | (n1 >> 11);
    const bool up2 = ((n1 >> 10) & 1u) && (((n1 & 0x3FFu) | n0 | nt) != 0 || (nl & 1u));
    const uint64_t nh = ((uint64_t)(n2 >> 11) << 32) | nl;
    lo = bitsd((((uint64_t)(uint32_t)(e - 53 - lz2 + 1022) << 52) + nh + (up2 ? 1 : 0)) |
               ((uint64_t)lneg << 63));
}

#undef BF_HD

}  // namespace bigf
}  // namespace mpdd
