// Device double-double arithmetic.
//
// A dd value is hi + lo with |lo| <= ulp(hi)/2 (the manual's dd format,
// Sec. 5: Knuth's TwoSum and Dekker's exact product on binary64).  Every
// operation here is written with the explicitly rounded intrinsics
// __dadd_rn / __dsub_rn / __dmul_rn / __fma_rn: the compiler never fuses or
// reassociates them, which the error-free transformations rely on (the
// manual's compiler note asks for the same: no value-changing FP
// optimisation for dd code).
#pragma once

namespace mpdd {

struct dd {
    double hi, lo;
};

// Rounded sum and difference: the intrinsics on the device, plain binary64
// on the host (where the check of two_sum compiles this header).
__host__ __device__ __forceinline__ double add_rn(double a, double b) {
#if defined(__CUDA_ARCH__)
    return __dadd_rn(a, b);
#else
    return a + b;
#endif
}
__host__ __device__ __forceinline__ double sub_rn(double a, double b) {
#if defined(__CUDA_ARCH__)
    return __dsub_rn(a, b);
#else
    return a - b;
#endif
}

// The leading 32 bits of |x|, shifted left by one: they order like the
// exponents of finite numbers, and like the magnitudes up to the trailing
// 32 significand bits.
__host__ __device__ __forceinline__ unsigned int lead_bits(double x) {
#if defined(__CUDA_ARCH__)
    return (unsigned int)__double2hiint(x) << 1;
#else
    unsigned long long u;
    __builtin_memcpy(&u, &x, 8);
    return (unsigned int)(u >> 32) << 1;
#endif
}

// TwoSum: s + e == a + b exactly, s = fl(a + b).  Knuth's form takes 6 FP64
// operations because it does not know which operand is the larger.  Here the
// leading words are compared and the operands exchanged on the integer pipe
// (7 instructions), after which Dekker's form needs 3: it is exact whenever
// the exponent of the first operand is at least that of the second.  e is the
// rounding error of s in either form, so the result is the same number bit
// for bit (the sign of a zero e aside; when s overflows, e is an infinity
// here and a NaN there, and the next renormalisation makes both NaN).
// An FP64 instruction occupies its partition of the SM for ~76 cycles and an
// integer one for 2, and every dd kernel is bound by the FP64 pipe: a dd
// multiply-add falls from 12.75 to 9.75 FP64 instructions, and the multiply-
// add mix of the plain kernel measured 85.9 before and 113.9 dd-GFlop/s now.
__host__ __device__ __forceinline__ void two_sum(double a, double b, double &s, double &e) {
    const bool swap = lead_bits(b) > lead_bits(a);
    const double big = swap ? b : a, small = swap ? a : b;
    s = add_rn(a, b);
    e = sub_rn(small, sub_rn(s, big));
}

// Dekker FastTwoSum (|a| >= |b| or a == 0): s + e == a + b.  3 operations.
__device__ __forceinline__ void fast_two_sum(double a, double b, double &s, double &e) {
    s = __dadd_rn(a, b);
    e = __dsub_rn(b, __dsub_rn(s, a));
}

// Product terms of a*b: p = fl(ah*bh), e = its exact error plus the two
// cross products ah*bl + al*bh (al*bl, below 2^-106 relative, is dropped).
// 1 DMUL + 3 DFMA.
__device__ __forceinline__ void prod_terms(dd a, dd b, double &p, double &e) {
    p = __dmul_rn(a.hi, b.hi);
    e = __fma_rn(a.hi, b.hi, -p);
    e = __fma_rn(a.hi, b.lo, e);
    e = __fma_rn(a.lo, b.hi, e);
}

// acc += (p + e), renormalised: TwoSum on the leading parts, the low parts
// added, FastTwoSum.  8 FP64 operations; absolute error at most ~2u^2
// (|acc| + |p|) per step (u = 2^-53).
__device__ __forceinline__ void acc_add(dd &acc, double p, double e) {
    double s, t;
    two_sum(acc.hi, p, s, t);
    t = __dadd_rn(t, __dadd_rn(acc.lo, e));
    fast_two_sum(s, t, acc.hi, acc.lo);
}

// One dd multiply-add: acc += a * b (12 FP64 operations).
__device__ __forceinline__ void mac(dd &acc, dd a, dd b) {
    double p, e;
    prod_terms(a, b, p, e);
    acc_add(acc, p, e);
}

// GEMM-loop multiply-add with deferred renormalisation: the leading parts
// are summed with TwoSum (exact), the TwoSum error and the product's low
// part are added into acc.lo, and the renormalisation is left until after
// every kRenormEvery steps of k (at l = 3, 7, 11, ... counted from the start of
// k, so every kernel renormalises at the same places): TwoSum in the GEMM
// kernels (renorm_mixed and renorm_exact, the same bits), FastTwoSum (renorm)
// in the Cholesky diagonal block and the 64-row solves.  4 + 3 + 2 = 9 FP64
// operations per step, 9.75 with the renormalisation (3 + 1 + 2 and 0.25 with
// the errors on the integer pipe).  Between renormalisations |acc.lo| stays within a few
// ulps of acc.hi, so each step's rounding error is at most ~(G+4) u^2
// (|acc| + |a b|) with G = 4: within the Rgemm bound 4 k 2^-104 (...).  A
// zero product leaves the state unchanged, so zero padding of k does not
// alter the result.
constexpr int kRenormEvery = 4;

// ---- the errors of a sum and of a product on the integer pipe
//
// The error of a sum or product that the FP64 pipe has rounded is a binary64
// number.  The FP64 pipe forms it with two more instructions (two_sum) or one
// (fma), each of which holds it for ~76 cycles of a warp; the integer pipe,
// idle beside it, forms it from the significands with ~60 or ~40 instructions
// of 2 cycles: modulo 2^64, because it is a small integer in the unit of the
// smaller operand's last place (of the product of the last places).  A dd
// multiply-add takes 6.25 FP64 instructions instead of 9.75: Rgemm 1101 x 700
// x 905 12.52 ms with none, 9.88 with the sum's error on the integer pipe,
// 8.73 with the product's as well, 8.08 with the renormalisation's; 512
// grouped problems 29.2, 23.0, 20.3 and 19.3 ms.
// The result is the same bits; the host compares both with the FP64 forms
// over the whole range in tests.

__host__ __device__ __forceinline__ unsigned long long bits_of(double x) {
#if defined(__CUDA_ARCH__)
    return (unsigned long long)__double_as_longlong(x);
#else
    unsigned long long u;
    __builtin_memcpy(&u, &x, 8);
    return u;
#endif
}
__host__ __device__ __forceinline__ double from_bits(unsigned long long u) {
#if defined(__CUDA_ARCH__)
    return __longlong_as_double((long long)u);
#else
    double x;
    __builtin_memcpy(&x, &u, 8);
    return x;
#endif
}

// A double's significand as an integer and the biased exponent of its last
// place's binade (1 for subnormals and zero): |x| = m 2^(e - 1075).
struct Significand {
    unsigned long long m;
    int e;
};
__host__ __device__ __forceinline__ Significand significand(unsigned long long u) {
    const unsigned int hi = (unsigned int)(u >> 32);
    const int f = (int)((hi >> 20) & 0x7FFu), normal = f < 1 ? f : 1;
    const unsigned int mh = (hi & 0xFFFFFu) + ((unsigned int)normal << 20);
    return Significand{((unsigned long long)mh << 32) | (unsigned int)u, f < 1 ? 1 : f};
}

// v times 2^(e - 1075) as a double with its sign exclusive-or'ed with bit 31
// of flip, for |v| < 2^53, e >= 1 and a result below the overflow threshold.
__host__ __device__ __forceinline__ double exact_double(long long v, int e, unsigned int flip) {
    const unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
#if defined(__CUDA_ARCH__)
    const int lead = __clzll((long long)a) - 11;
#else
    const int lead = (a ? __builtin_clzll(a) : 64) - 11;
#endif
    // the leading one at bit 52 adds one to the exponent field below it; where
    // the exponent does not reach that far, the field is zero (subnormal)
    const int n = lead < e - 1 ? lead : e - 1;
    const unsigned long long r =
        (a << (n & 63)) + ((unsigned long long)(unsigned int)(e - n - 1) << 52);
    const unsigned long long sign =
        (unsigned long long)((v < 0 ? 0x80000000u : 0u) ^ flip) << 32;
    return a == 0 ? 0.0 : from_bits(r | sign);
}

// x + y - s for s = RN(x + y), NaN where s is an infinity or NaN.  With B the
// larger, S the smaller and d the difference of their exponents, 2 (B - s) is
// an integer of at most 55 bits in half units of B's last place (s is at most
// one binade off B, or the sum is exact); d binades down and S added, it is
// twice the error in units of S's last place.  Where s is B, the error is S:
// that covers every d above 54.
// Subnormals and non-finite numbers are part of the integer form on purpose:
// with a branch to the FP64 form for them the compiler predicates the two FP64
// instructions, which then hold the pipe in every step.
__host__ __device__ __forceinline__ double sum_error(double x, double y, double s) {
    const unsigned long long ux = bits_of(x), uy = bits_of(y), us = bits_of(s);
    const bool swap = lead_bits(y) > lead_bits(x);
    const unsigned long long B = swap ? uy : ux, S = swap ? ux : uy;
    const unsigned int Bh = (unsigned int)(B >> 32), Sh = (unsigned int)(S >> 32);
    const Significand mB = significand(B), mS = significand(S), ms = significand(us);
    const int k = ms.e - mB.e + 1;   // 0, 1, 2; below: the sum is exact
    const unsigned long long D = (mB.m << 1) - (ms.m << (k & 3));
    const unsigned long long t = mS.m << 1;
    const unsigned long long E =
        (D << ((mB.e - mS.e) & 63)) + (((Bh ^ Sh) >> 31) ? 0ull - t : t);
    double e = exact_double((long long)E >> 1, mS.e, Bh & 0x80000000u);
    const int other_sign = (int)((unsigned int)(us >> 32) ^ Bh);   // B and S of one leading word
    e = us == B ? from_bits(S) : (k | other_sign) < 0 ? 0.0 : e;
    return ms.e == 0x7FF ? from_bits(0x7FF8000000000000ull) : e;
}

// a b - p for p = RN(a b): fma(a, b, -p) from the integer pipe (the sign of a
// zero aside; NaN where p is an infinity or NaN).  The significands' product
// and p's agree above the unit 2^52 or 2^53 of p, so the low 64 bits of the
// one minus the other are the error as an integer of at most 53 bits.  A p
// below 2^-1021 has an error of half a subnormal unit at most, which rounds to
// zero; so has one that subnormal factors leave exact.
__host__ __device__ __forceinline__ double prod_error(double a, double b, double p) {
    const unsigned long long ua = bits_of(a), ub = bits_of(b);
    const Significand ma = significand(ua), mb = significand(ub), mp = significand(bits_of(p));
    int e0 = ma.e + mb.e - 1075;   // the unit of the product is 2^(e0 - 1075)
    const int sh = mp.e - e0;
    long long v = (long long)(ma.m * mb.m - (mp.m << (sh & 63)));
    if (e0 < 1) {   // the error's last places lie below the subnormals: round to even
        const int t = 1 - e0 > 54 ? 54 : 1 - e0;
        const unsigned long long w = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
        const unsigned long long q = (w + ((1ull << (t - 1)) - 1) + ((w >> t) & 1)) >> t;
        v = v < 0 ? -(long long)q : (long long)q;
        e0 = 1;
    }
    double e = exact_double(v, e0, (unsigned int)((ua ^ ub) >> 32) & 0x80000000u);
    e = (mp.e <= 1 || sh < 0) ? 0.0 : e;
    return mp.e == 0x7FF ? from_bits(0x7FF8000000000000ull) : e;
}

__device__ __forceinline__ void mac_deferred(dd &acc, dd a, dd b) {
    double p, e, s, e1;
    prod_terms(a, b, p, e);
    two_sum(acc.hi, p, s, e1);
    acc.hi = s;
    acc.lo = __dadd_rn(acc.lo, __dadd_rn(e1, e));
}

// mac_deferred with both errors from the integer pipe: the same result.
__device__ __forceinline__ void mac_mixed(dd &acc, dd a, dd b) {
    const double p = __dmul_rn(a.hi, b.hi);
    const double e = __fma_rn(a.lo, b.hi, __fma_rn(a.hi, b.lo, prod_error(a.hi, b.hi, p)));
    const double s = __dadd_rn(acc.hi, p);
    const double e1 = sum_error(acc.hi, p, s);
    acc.hi = s;
    acc.lo = __dadd_rn(acc.lo, __dadd_rn(e1, e));
}

// The GEMM kernels' renormalisation: TwoSum, exact whatever cancellation has
// left in hi, with the error from the integer pipe (one FP64 instruction
// instead of FastTwoSum's three) or, the same bits, from the FP64 pipe.
__device__ __forceinline__ void renorm_mixed(dd &acc) {
    const double s = __dadd_rn(acc.hi, acc.lo);
    acc.lo = sum_error(acc.hi, acc.lo, s);
    acc.hi = s;
}
__device__ __forceinline__ void renorm_exact(dd &acc) { two_sum(acc.hi, acc.lo, acc.hi, acc.lo); }

__device__ __forceinline__ void renorm(dd &acc) { fast_two_sum(acc.hi, acc.lo, acc.hi, acc.lo); }

// dd product, renormalised.
__device__ __forceinline__ dd mul(dd a, dd b) {
    double p, e;
    prod_terms(a, b, p, e);
    dd r;
    fast_two_sum(p, e, r.hi, r.lo);
    return r;
}

// Accurate dd addition (two TwoSums, two renormalisations): relative error
// at most 3u^2 + 13u^3.
__device__ __forceinline__ dd add(dd a, dd b) {
    double s1, s2, t1, t2;
    two_sum(a.hi, b.hi, s1, s2);
    two_sum(a.lo, b.lo, t1, t2);
    s2 = __dadd_rn(s2, t1);
    fast_two_sum(s1, s2, s1, s2);
    s2 = __dadd_rn(s2, t2);
    dd r;
    fast_two_sum(s1, s2, r.hi, r.lo);
    return r;
}

// Sloppy dd addition (TwoSum on the leading parts, low parts added,
// FastTwoSum): 8 FP64 operations, absolute error at most ~2u^2 (|a| + |b|)
// (the relative error can be large under cancellation).  Used where the
// accuracy target is the absolute bound 4 k 2^-104 (|alpha||A||B| +
// |beta||C|), e.g. the final alpha/beta combination.
__device__ __forceinline__ dd add_sloppy(dd a, dd b) {
    double s, e;
    two_sum(a.hi, b.hi, s, e);
    e = __dadd_rn(e, __dadd_rn(a.lo, b.lo));
    dd r;
    fast_two_sum(s, e, r.hi, r.lo);
    return r;
}

__device__ __forceinline__ dd neg(dd a) { return dd{-a.hi, -a.lo}; }
__device__ __forceinline__ dd sub(dd a, dd b) { return add(a, neg(b)); }

// dd division by two steps of long division.  q1 = RN(a.hi / b.hi); the
// remainder of a correctly rounded quotient, a.hi - q1 b.hi, is a binary64
// number, so one FMA gives it exactly; the rest of a - q1 b (a.lo - q1 b.lo)
// is added with two roundings, and q2 = RN(remainder / b.hi).  Relative
// error at most ~11 u^2 (u = 2^-53).  When a and b are binary64 numbers
// (a.lo = b.lo = 0) whose quotient is one too, q1 is that quotient, the
// remainder is 0 and the result exact.  The dependent chain is two
// divisions and five FP64 operations: this is what the row-serial
// triangular solves and the Cholesky pivots wait on.
__device__ __forceinline__ dd div(dd a, dd b) {
    const double q1 = __ddiv_rn(a.hi, b.hi);
    double r = __fma_rn(-q1, b.hi, a.hi);
    r = __dadd_rn(r, __fma_rn(-q1, b.lo, a.lo));
    const double q2 = __ddiv_rn(r, b.hi);
    dd q;
    fast_two_sum(q1, q2, q.hi, q.lo);
    return q;
}

// The exponent field of x lies in [128, 1918] (2^-895 to 2^896): its parts
// 2^-106 below it and its reciprocal are normal.
__device__ __forceinline__ bool mid_range(double x) {
    return (((unsigned int)__double2hiint(x) >> 20) & 0x7FFu) - 128u <= 1790u;
}

// a / b for binary64 numbers from y, an approximation of 1 / b within a few
// ulps: q0 = RN(a y) is within a few ulps of a / b, and the remainder a - q0 b
// (one FMA) times y corrects it, so the result is a / b rounded once, but for
// near-ties, and a / b itself whenever that is a binary64 number (Markstein,
// "Computation of elementary functions on the IBM RISC System/6000
// processor", 1990), as long as a / b is normal.  Operands of opposite extremes
// are not singled out: where a / b is below the normal range the result is
// within a subnormal unit of it, and where it overflows the result is a NaN
// (which the remainder makes of div_rcp's quotient in any case).  Three FP64
// instructions on the dependent chain, where the division takes as long as nine
// (576 cycles of a warp).  Operands near the ends of the exponent range, zeros
// and non-finite ones are divided.
__device__ __forceinline__ double quotient(double a, double b, double y) {
    if (!(mid_range(a) && mid_range(b))) return __ddiv_rn(a, b);
    const double q = __dmul_rn(a, y);
    return __fma_rn(__fma_rn(-q, b, a), y, q);
}

// dd division with a given approximate reciprocal y of b.hi (within a few
// ulps): div's long division with both quotient digits taken by y, so the
// dependent chain holds no division.  The second digit's extra relative error
// (a few u) is scaled by |q2| <= ~3u |a / b|: the result's relative error stays
// at most ~20 u^2, and an exactly representable quotient of binary64
// operands is still exact (its remainder is 0).  a need not be
// renormalised: |a.lo| may be a few ulps of a.hi.
__device__ __forceinline__ dd div_rcp(dd a, dd b, double y) {
    const double q1 = quotient(a.hi, b.hi, y);
    double r = __fma_rn(-q1, b.hi, a.hi);
    r = __dadd_rn(r, __fma_rn(-q1, b.lo, a.lo));
    const double q2 = __dmul_rn(r, y);
    dd q;
    fast_two_sum(q1, q2, q.hi, q.lo);
    return q;
}

// dd reciprocal 1 / b: div(1, b) with the first digit RN(1 / b.hi) from
// the correctly rounded reciprocal (the same number as the division gives)
// and the second taken by it as well: one reciprocal, five FP64 operations.
__device__ __forceinline__ dd rcp_dd(dd b) {
    const double y = __drcp_rn(b.hi);
    double r = __fma_rn(-y, b.hi, 1.0);
    r = __fma_rn(-y, b.lo, r);
    dd q;
    fast_two_sum(y, __dmul_rn(r, y), q.hi, q.lo);
    return q;
}

// dd square root: x = sqrt(a.hi) rounded, whose remainder a.hi - x^2 is a
// binary64 number (one FMA gives it exactly), plus one Newton correction
// (a - x^2) / (2x) with a.lo added, the division taken as a product with
// z = rsqrt(a.hi) (1 ulp); the neglected second-order term is below u^2 / 8
// relative.  x is x0 = RN(a.hi z) corrected once by its own remainder,
// x0 + (a.hi - x0^2) z / 2: sqrt(a.hi) rounded once but for near-ties, and the
// root itself when that is a binary64 number (the same method as quotient);
// near the ends of the exponent range the square root is taken.  Exact when
// a.hi is the square of a binary64 number and a.lo = 0.  z, an approximate
// reciprocal of the result's leading part within a few ulps, is returned for
// div_rcp.  a need not be renormalised.  Returns 0 (and z = 0) for a <= 0.
__device__ __forceinline__ dd sqrt_dd(dd a, double &z) {
    z = 0.0;
    if (!(a.hi > 0.0)) return dd{0.0, 0.0};
    z = rsqrt(a.hi);
    const double hz = __dmul_rn(z, 0.5);
    double x;
    if (mid_range(a.hi)) {
        const double x0 = __dmul_rn(a.hi, z);
        x = __fma_rn(__fma_rn(-x0, x0, a.hi), hz, x0);
    } else {
        x = __dsqrt_rn(a.hi);
    }
    const double r = __dadd_rn(__fma_rn(-x, x, a.hi), a.lo);
    dd s;
    fast_two_sum(x, __dmul_rn(r, hz), s.hi, s.lo);
    return s;
}

}  // namespace mpdd
