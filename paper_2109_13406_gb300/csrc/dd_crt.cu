// Residue (CRT) form of the split-precision dd Rgemm on the fp16 tensor cores.
//
// The exact integers of the sliced form at a width of W = 8D bits --
// X = RNE(hi 2^(W - e)) + RNE(lo 2^(W - e)) for an entry x = hi + lo of a row
// of op(A) with scale e (and likewise for the columns of op(B)),
// |X| < 2^(W-1) -- are multiplied exactly through the Chinese remainder
// theorem instead of through digit pairs:
//
//  1. residues: r_i = X mod p_i in the symmetric range (|r_i| <= 128) for
//     N pairwise coprime moduli p_i <= 256, stored as exact fp16 planes;
//  2. products: C_i = R^A_i (R^B_i)^T on the tensor cores with the exact
//     fp32-run / int32 accumulation of the band kernel (diagonal mode), each
//     stored reduced mod p_i (one byte);
//  3. reconstruction: C' = sum_i c_i w_i mod P with P = prod p_i and the CRT
//     weights w_i = (P/p_i) ((P/p_i)^-1 mod p_i), in multiword integer
//     arithmetic, mapped to the symmetric range; since P >= k 2^(2W) >
//     4 |A' B'|, C' is exactly the integer product A'B'; it is rounded once
//     to dd, scaled by 2^(e_i + f_j - 2W), and alpha/beta are applied in dd.
//
// The only error is the rounding of A and B to W bits: at most
// (1 + 2^-W) 2^(e_i + f_j - W) per product.  Each call certifies it against
// the accuracy bound before choosing W (ozaki_common.cuh): 112 bits (D = 14
// digits, 32 moduli at k = 8192) when that suffices, else 120 or 128 bits
// (more moduli), else the plain FP64 kernel computes the product.  N is the
// smallest even count with P >= k 2^(2W), against S(S+1)/2 = 105 pair
// products of the 14-digit sliced form at W = 112.
#include <cuda_fp16.h>

#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include "bigfloat.cuh"
#include "common.cuh"
#include "dd_arith.cuh"
#include "kernels.cuh"
#include "ozaki_common.cuh"

namespace mpdd {
namespace {

constexpr int kMinDigits = 14;        // X has D base-256 digits, W = 8 D bits
constexpr int kMaxDigits = 16;        // |X| < 2^127: a signed 128-bit integer
constexpr int kMaxMod = 40;
constexpr int kWords = 11;           // 32-bit words for sums below 2^352
// pairwise coprime moduli <= 256, largest first: 2^8, 3*5*17, 11*23, 13*19
// and primes not dividing those
__host__ __device__ constexpr int modulus(int i) {
    constexpr int m[kMaxMod] = {256, 255, 253, 251, 247, 241, 239, 233, 229, 227,
                                223, 211, 199, 197, 193, 191, 181, 179, 173, 167,
                                163, 157, 151, 149, 139, 137, 131, 127, 113, 109,
                                107, 103, 101, 97,  89,  83,  79,  73,  71,  67};
    return m[i];
}

// 256^t mod p_b.
__host__ __device__ constexpr int pow256_mod(int t, int b) {
    int v = 1 % modulus(b);
    for (int u = 0; u < t; ++u) v = (v * 256) % modulus(b);
    return v;
}

// The fp16 bits of an integer in [0, 255] (exact).
__host__ __device__ constexpr unsigned half_bits(int v) {
    if (v == 0) return 0u;
    int e = 0;
    while ((v >> (e + 1)) != 0) ++e;
    return ((unsigned)(e + 15) << 10) | (((unsigned)v << (10 - e)) & 0x3FFu);
}

// Residues on the tensor cores.  For an entry X (the scaled integer of
// RNE(hi 2^s) + RNE(lo 2^s), |X| < 2^(8D-1) for D digit bytes) the biased
// X' = X + 2^(8D-1) has D unsigned bytes x_t, and
//     s_b = sum_t x_t (256^t mod p_b) - (2^(8D-1) mod p_b)
// is congruent to X mod p_b with -255 <= s_b < 16 255^2 < 2^22.  Over 16
// entries the sums are the product [16 entries x 16 bytes] x [16 bytes x 8
// moduli], done by mma.sync m16n8k16: a byte is the fp16 1024 + x_t (exact)
// and the fp32 accumulator of modulus b starts at -1024 sum_t (256^t mod
// p_b) - (2^(8D-1) mod p_b), so it ends at exactly s_b (every partial sum an
// integer below 2^23 in magnitude).  r = s - p rint(s / p) is then the
// residue in [-(p-1)/2, (p-1)/2] for odd p: the fp32 quotient is within
// |s / p| 2^-23 of s / p, below 1 / (2 p), while s / p, an integer over an
// odd p, is never within 1 / (2 p) of a half-integer.  For p = 256 the
// lowest byte of X, taken in [-128, 127], is the residue.  Moduli 1 .. N-1
// sit in n-tiles of 8; the first N planes are written (N and D from the
// call's certificate).
//
// A warp computes 64 consecutive k of one row.  Each lane forms X' of two
// entries and leaves its words in shared memory, from where lane (g, q) of the
// warp's quads takes the bytes 2q, 2q+1, 2q+8, 2q+9 of the entries 8g .. 8g+7
// (the A fragments of four m16 tiles); its accumulators then hold two moduli
// of those eight consecutive k, stored as one 16-byte write per modulus (a
// whole 128-byte line per modulus and warp).  Rows that are contiguous in
// memory reach a block as a 16 x 64 tile, read along the rows and turned in
// shared memory, so both layouts share the rest; the next entries are loaded
// before the present ones are computed.  Both operands of a call go in one
// launch of as many blocks as are resident.
//
// What bounds it: 16 bytes read and 64 written per entry (1.58 ms of HBM time
// for both operands of an 8192 product) against instruction issue and the
// shared-memory wavefronts of the tables (32 k per warp and 8-byte stores ran
// the wavefronts at 74 % of their peak; they are at 84 % now).  Both operands of
// an 8192 product: 2.03 ms, 0.78 of the copy rate; an FP32 kernel for the
// row-contiguous operand and this one with 128-bit shifts left to the
// compiler and a byte exchange by shuffles took 3.44 ms.
constexpr int kResNT = (kMaxMod - 1 + 7) / 8;   // n-tiles of moduli 1 .. 39
constexpr int kResThreads = 256, kResWarps = kResThreads / 32, kResBlocks = 3;

// D = A B + C for one m16n8k16 tile: fp16 A (row) and B (col), fp32 C / D.
__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint2 b,
                                          const float (&c)[4]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%10,%11,%12,%13};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y), "f"(c[0]), "f"(c[1]),
          "f"(c[2]), "f"(c[3]));
}

struct alignas(16) ResLane {   // per n-tile and lane: B fragment, accumulator starts,
    unsigned b0, b1;           // and the reduction constants of the lane's 2 moduli
    float init0, init1;
    float inv[2], negp[2];     // {1/p0, 1/p1}, {-p0, -p1}
};

// For D = 14, 15, 16 digit bytes; the moduli past a call's N are computed
// with the others and not stored.
struct ResTables {
    ResLane t[kMaxDigits - kMinDigits + 1][kResNT * 32];
};

constexpr ResTables make_res_tables() {
    ResTables T{};
    for (int D = kMinDigits; D <= kMaxDigits; ++D)
        for (int nt = 0; nt < kResNT; ++nt)
            for (int lane = 0; lane < 32; ++lane) {
                const int g = lane >> 2, q = lane & 3;
                ResLane L{};
                const int bm = 1 + 8 * nt + g;   // B column g
                auto h = [&](int t) {
                    return bm < kMaxMod && t < D ? half_bits(pow256_mod(t, bm)) : 0u;
                };
                L.b0 = h(2 * q) | (h(2 * q + 1) << 16);
                L.b1 = h(2 * q + 8) | (h(2 * q + 9) << 16);
                float init[2] = {0.0f, 0.0f};
                for (int e = 0; e < 2; ++e) {
                    const int m = 1 + 8 * nt + 2 * q + e;   // C column 2q + e
                    if (m >= kMaxMod) continue;
                    int ws = 0;
                    for (int t = 0; t < D; ++t) ws += pow256_mod(t, m);
                    const int bias = (128 * pow256_mod(D - 1, m)) % modulus(m);
                    init[e] = (float)(-1024 * ws - bias);   // exact: below 2^23
                    L.inv[e] = 1.0f / (float)modulus(m);
                    L.negp[e] = -(float)modulus(m);
                }
                L.init0 = init[0];
                L.init1 = init[1];
                T.t[D - kMinDigits][nt * 32 + lane] = L;
            }
    return T;
}

__device__ const ResTables g_res_tables = make_res_tables();

struct ResOperand {
    const double *hi, *lo;
    int64_t ld;
    int row_contig;
    int64_t rows, rows_pad;
    const unsigned long long *max;
    __half *R;
    unsigned blocks;   // its blocks of the launch
};

struct ResShared {
    ResLane tab[kResNT * 32];
    // words (0, 2, 1, 3) of the warp's 64 integers, eight to a row of 36
    // words: 16-byte stores and 8-byte reads without bank conflicts
    uint32_t x[kResWarps][8 * 36];
    double hi[64][17], lo[64][17];   // row-contiguous tiles, [l][row]
};

// Residues of the 64 entries (row, 64 c + lane) and (row, 64 c + 32 + lane)
// from the lane's two X'; base: the address of plane 0's entry (row, 64 c + 8
// g), ps: entries of a plane.
__device__ __forceinline__ void residue_warp(const unsigned __int128 (&Xb)[2], __half *base,
                                             int64_t ps, int N, const ResLane *tab,
                                             uint32_t *xw) {
    const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
    const float2 magic{12582912.0f, 12582912.0f}, nmagic{-12582912.0f, -12582912.0f};
    __syncwarp();   // the previous entries' words have been read
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int at = lane + 32 * u;
        *reinterpret_cast<uint4 *>(xw + (at >> 3) * 36 + (at & 7) * 4) =
            make_uint4((uint32_t)Xb[u], (uint32_t)(Xb[u] >> 64), (uint32_t)(Xb[u] >> 32),
                       (uint32_t)(Xb[u] >> 96));
    }
    __syncwarp();
    // A fragments of tile t: row g = entry 8g + 2t, row g + 8 = entry 8g + 2t + 1,
    // each byte as the fp16 1024 + x
    const uint32_t sel = (q & 1) ? 0x4342u : 0x4140u;
    uint32_t A[4][4];
    uint32_t low[4] = {0u, 0u, 0u, 0u};   // the lowest bytes of the entries, lane q = 0
#pragma unroll
    for (int t = 0; t < 4; ++t)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            // words q/2 and 2 + q/2 of the entry
            const uint2 w = *reinterpret_cast<const uint2 *>(xw + g * 36 + (2 * t + h) * 4 +
                                                             (q >> 1) * 2);
            A[t][h] = __byte_perm(w.x, 0x64646464u, sel);
            A[t][2 + h] = __byte_perm(w.y, 0x64646464u, sel);
            low[t] |= (w.x & 0xFFu) << (16 * h);
        }
    // plane 0 (p = 256): the lowest byte x of X, signed: with its top bit
    // turned, fp16 1024 + (x ^ 128) less 1152
    if (q == 0) {
        uint32_t o[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const uint32_t b = (low[t] ^ 0x00800080u) | 0x64006400u;
            const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&b),
                                      __floats2half2_rn(1152.0f, 1152.0f));
            o[t] = *reinterpret_cast<const uint32_t *>(&h);
        }
        *reinterpret_cast<uint4 *>(base) = make_uint4(o[0], o[1], o[2], o[3]);
    }
    __half *dst = base + (1 + 2 * q) * ps;
#pragma unroll
    for (int nt = 0; nt < kResNT; ++nt, dst += 8 * ps) {
        if (1 + 8 * nt >= N) break;
        const ResLane &L = tab[nt * 32 + lane];
        const float4 start = *reinterpret_cast<const float4 *>(&L.b0);
        const float4 red = *reinterpret_cast<const float4 *>(L.inv);
        const float2 iv{red.x, red.y}, np{red.z, red.w};
        const float c0[4] = {start.z, start.w, start.z, start.w};
        const uint2 bf = make_uint2(__float_as_uint(start.x), __float_as_uint(start.y));
        uint32_t o0[4], o1[4];   // the lane's two moduli, entries 2t and 2t + 1
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            float acc[4];
            mma_16816(acc, A[t], bf, c0);
            float2 r[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float2 s2{acc[2 * h], acc[2 * h + 1]};
                const float2 qn = __fadd2_rn(__ffma2_rn(s2, iv, magic), nmagic);
                r[h] = __ffma2_rn(np, qn, s2);
            }
            const __half2 h0 = __floats2half2_rn(r[0].x, r[1].x);
            const __half2 h1 = __floats2half2_rn(r[0].y, r[1].y);
            o0[t] = *reinterpret_cast<const uint32_t *>(&h0);
            o1[t] = *reinterpret_cast<const uint32_t *>(&h1);
        }
        if (1 + 8 * nt + 2 * q < N)
            *reinterpret_cast<uint4 *>(dst) = make_uint4(o0[0], o0[1], o0[2], o0[3]);
        if (2 + 8 * nt + 2 * q < N)
            *reinterpret_cast<uint4 *>(dst + ps) = make_uint4(o1[0], o1[1], o1[2], o1[3]);
    }
}

// X + 2^(8 DG - 1) of a dd entry at scale e.  The lo part of a normalised dd
// at 112 bits is below 2^59: 64-bit arithmetic, whenever that holds.
__device__ __forceinline__ unsigned __int128 biased_integer(double hi, double lo, int DG, int e) {
    const int shift = 8 * DG - e;
    const int E = (int)(((uint32_t)__double2hiint(lo) >> 20) & 0x7FF);
    __int128 L;
    if (E - 1075 + shift <= 9) {   // |lo 2^shift| < 2^62
        const unsigned long long bits = (unsigned long long)__double_as_longlong(lo);
        unsigned long long m =
            (bits & ((1ull << 52) - 1)) | ((unsigned long long)(E ? 1 : 0) << 52);
        const int sh = (E ? E : 1) - 1075 + shift;
        if (sh < 0) {
            const int rs = -sh < 60 ? -sh : 60;
            m = (m + ((1ull << (rs - 1)) - 1) + ((m >> rs) & 1)) >> rs;
        } else {
            m <<= sh;
        }
        const long long v = (long long)m;
        L = (bits >> 63) ? -v : v;
    } else {
        L = scaled_round(lo, shift);
    }
    return (unsigned __int128)(scaled_round(hi, shift) + L) +
           ((unsigned __int128)1 << (8 * DG - 1));
}

__global__ void __launch_bounds__(kResThreads, kResBlocks) residue_kernel(
    const ResOperand a, const ResOperand b, int64_t k, int64_t k_pad, const SplitPlan plan) {
    __shared__ ResShared sh;
    chain_begin();
    const PlanPick pk = plan_choice(plan);
    if (pk.c < 0) return;
    const int N = pk.count, DG = pk.width / 8;
    const bool first = blockIdx.x < a.blocks;
    const double *Xh = first ? a.hi : b.hi, *Xl = first ? a.lo : b.lo;
    const int64_t ld = first ? a.ld : b.ld, rows = first ? a.rows : b.rows;
    const int64_t rows_pad = first ? a.rows_pad : b.rows_pad;
    const int row_contig = first ? a.row_contig : b.row_contig;
    const unsigned long long *rmax = first ? a.max : b.max;
    __half *R = first ? a.R : b.R;
    const unsigned bid = first ? blockIdx.x : blockIdx.x - a.blocks;
    const unsigned nblk = first ? a.blocks : b.blocks;
    for (int x = threadIdx.x; x < kResNT * 32; x += kResThreads)
        sh.tab[x] = g_res_tables.t[DG - kMinDigits][x];
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x / 32;
    const int64_t ps = rows_pad * k_pad;
    const int64_t cols = k_pad / 64;             // 64-entry chunks of a row
    uint32_t *xw = sh.x[warp];
    // items in order, chunk fastest: (row, chunk) per warp, or (16 rows,
    // chunk) per block; the stride is kept as whole rows and a remainder
    const int64_t stride = row_contig ? (int64_t)nblk : (int64_t)nblk * kResWarps;
    const int64_t start = row_contig ? (int64_t)bid : (int64_t)bid * kResWarps + warp;
    const int64_t end = row_contig ? rows_pad / 16 : rows_pad;
    int64_t i = start / cols, c = start - i * cols;
    const int64_t si = stride / cols, sc = stride - si * cols;
    if (!row_contig) {
        double hi[2], lo[2];
        int e = 0;
        auto fetch = [&](int64_t row, int64_t ch) {
            const int64_t l = 64 * ch + lane;
            const double *ph = Xh + l + row * ld, *pl = Xl + l + row * ld;
            e = 0;
            if (row < rows) e = scale_exponent(__ldg(rmax + row));
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const bool ok = row < rows && l + 32 * u < k;
                hi[u] = ok ? __ldg(ph + 32 * u) : 0.0;
                lo[u] = ok ? __ldg(pl + 32 * u) : 0.0;
            }
        };
        if (i < end) fetch(i, c);
        while (i < end) {
            const unsigned __int128 Xb[2] = {biased_integer(hi[0], lo[0], DG, e),
                                             biased_integer(hi[1], lo[1], DG, e)};
            __half *base = R + i * k_pad + 64 * c + 8 * (lane >> 2);
            i += si;
            c += sc;
            if (c >= cols) {
                c -= cols;
                ++i;
            }
            if (i < end) fetch(i, c);
            residue_warp(Xb, base, ps, N, sh.tab, xw);
        }
        return;
    }
    double fh[4], fl[4];
    const int tr = threadIdx.x % 16, tl = threadIdx.x / 16;
    auto fetch = [&](int64_t rt, int64_t ch) {
        const int64_t row = 16 * rt + tr;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t l = 64 * ch + tl + 16 * u;
            const bool ok = row < rows && l < k;
            fh[u] = ok ? __ldg(Xh + row + l * ld) : 0.0;
            fl[u] = ok ? __ldg(Xl + row + l * ld) : 0.0;
        }
    };
    if (i < end) fetch(i, c);
    while (i < end) {
        __syncthreads();   // the previous tile has been read
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            sh.hi[tl + 16 * u][tr] = fh[u];
            sh.lo[tl + 16 * u][tr] = fl[u];
        }
        __syncthreads();
        const int64_t ti = i, tc = c;
        i += si;
        c += sc;
        if (c >= cols) {
            c -= cols;
            ++i;
        }
        if (i < end) fetch(i, c);
#pragma unroll 1
        for (int u = 0; u < 2; ++u) {
            const int rr = warp + kResWarps * u;
            const int64_t row = 16 * ti + rr;
            const int e = row < rows ? scale_exponent(__ldg(rmax + row)) : 0;
            const unsigned __int128 Xb[2] = {
                biased_integer(sh.hi[lane][rr], sh.lo[lane][rr], DG, e),
                biased_integer(sh.hi[lane + 32][rr], sh.lo[lane + 32][rr], DG, e)};
            residue_warp(Xb, R + row * k_pad + 64 * tc + 8 * (lane >> 2), ps, N, sh.tab, xw);
        }
    }
}

// ------------------------------------------------------------------ CRT

// Reconstruction constants of one moduli count N.
struct CrtTables {
    // Byte t of the CRT weights w_b = (P / p_b) ((P / p_b)^-1 mod p_b) of the
    // four moduli b = 4g .. 4g+3, packed in one word (zero past N): the dp4a
    // operand of digit t of the sums.
    uint32_t wp[kMaxMod / 4][4 * kWords];
    // Byte t of qfix_b = RN(2^24 ((P / p_b)^-1 mod p_b) / p_b), w_b / P in
    // fixed point, of the moduli b = 4g .. 4g+3.
    uint32_t qp[kMaxMod / 4][3];
    // 16-bit digits of 2^(32 kWords) - P, P the product of the moduli.
    uint32_t negp[2 * kWords];
};

struct CrtArgs {
    SplitPlan plan;                       // N and W of the call (tab[c] for candidate c)
    CrtTables tab[kMaxCand];
    int64_t m, n, m_pad, n_pad;
    const uint8_t *res;                   // [N][n_pad][m_pad] products mod p_i
    const unsigned long long *rmax, *cmax;
    mp_dd alpha, beta;
    int alpha_one, beta_zero;
    int ab_mode;                          // 0 general; alpha = +-1 and beta = 0 (1) or 1 (2);
                                          // 3 (updates): alpha = +-1, general beta
    int alpha_neg;                        // alpha = -1 (modes 1 to 3)
    double *ch, *cl;
    int64_t ldc;
    int tri;                              // 0: all of C; 1 / 2: upper / lower triangle
    int single;                           // one entry per thread, no loop
    const int64_t *info;                  // optional: non-zero -> leave C as is
};

// alpha v + beta c in dd with one rounding chain: the two leading products
// split exactly (product and FMA error), their sum by TwoSum, every
// lower-order term added into the error word, one FastTwoSum.  Absolute error
// within about 3u^2 (|alpha v| + |beta c|), u = 2^-53; 17 FP64 operations
// against 22 for two dd products and a dd sum.
__device__ __forceinline__ dd axpby_dd(dd alpha, dd v, dd beta, dd c) {
    const double p1 = __dmul_rn(alpha.hi, v.hi), e1 = __fma_rn(alpha.hi, v.hi, -p1);
    const double p2 = __dmul_rn(beta.hi, c.hi), e2 = __fma_rn(beta.hi, c.hi, -p2);
    double s, t;
    two_sum(p1, p2, s, t);
    const double low = __fma_rn(alpha.hi, v.lo,
                                __fma_rn(alpha.lo, v.hi, __fma_rn(beta.hi, c.lo,
                                                                  __dmul_rn(beta.lo, c.hi))));
    t = __dadd_rn(t, __dadd_rn(__dadd_rn(e1, e2), low));
    dd r;
    fast_two_sum(s, t, r.hi, r.lo);
    return r;
}

// The reconstructed integer of one entry from its N products reduced mod p_b
// (four to a register): Z = sum_b c_b w_b - q P over NW 32-bit words in two's
// complement.  q is the integer nearest to S / P = sum_b c_b (inv_b / p_b),
// S = sum_b c_b w_b: |Z| < k 2^(2W-2) <= P / 4 puts S / P at least 1/4 from a
// half-integer, while the fixed-point column (each qfix_b within 2^-25 of
// inv_b / p_b, 16 bits of the sum kept) is within N 255 2^-25 + 2^-15 <
// 0.0005 of it.  Then each byte digit of S is a column summed by one dp4a per
// four moduli (below 40 255^2 < 2^22), two columns and q times the 16-bit
// digit of -P make a half word (below 2^31), and one carry runs up the words.
// T is a reference into the kernel's parameter block: its words are
// constant-bank operands.  (16-bit columns with dp2a, half as many to carry,
// were slower: the constant has to be dp2a's 16-bit operand, which the
// instruction does not read from the constant bank.)
//
// What bounds the kernel: the ~17 FP64 operations of a general alpha / beta
// epilogue (2.15 ms at 8192 x 8192), beside ~330 multiply-add-class integer
// instructions at 64 lanes per clock and SM (1.1 ms) and as many issue slots
// of others.  A separate subtraction of q P, a full negation and general
// 128-bit shifts made ~1120 instructions per entry (747 now): at 8192 x 8192
// 3.43 ms before and 2.42 now with general alpha and beta, 2.83 and 1.63 with
// alpha = 1 and beta = 0.
template <int NW, int G>
__device__ __forceinline__ void crt_integer(const CrtTables &T, const uint32_t (&R)[G],
                                            uint32_t (&Z)[NW]) {
    uint32_t q0 = 0, q1 = 0, q2 = 0;
#pragma unroll
    for (int g = 0; g < G; ++g) {
        q0 = __dp4a(R[g], T.qp[g][0], q0);
        q1 = __dp4a(R[g], T.qp[g][1], q1);
        q2 = __dp4a(R[g], T.qp[g][2], q2);
    }
    const uint32_t q = ((q0 >> 8) + q1 + (q2 << 8) + (1u << 15)) >> 16;
    uint32_t c = 0;
#pragma unroll
    for (int t = 0; t < NW; ++t) {
        uint32_t d[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int g = 0; g < G; ++g) {
#pragma unroll
            for (int u = 0; u < 4; ++u) d[u] = __dp4a(R[g], T.wp[g][4 * t + u], d[u]);
        }
        const uint32_t x = q * T.negp[2 * t] + (d[1] * 256u + d[0]);
        const uint32_t y = q * T.negp[2 * t + 1] + (d[3] * 256u + d[2]);
        // word t: x + 2^16 y + the carry (below 2^31 + 2^16 + 2^47)
        const uint64_t v = (uint64_t)y * 65536u + (x + c);
        Z[t] = (uint32_t)v;
        c = (uint32_t)(v >> 32);
    }
}

// The alpha / beta epilogue of one entry: v its product, (ch, cl) the old C
// where the epilogue reads it.  UPD (a solve's or factorisation's update, which
// takes a solve's alpha as its beta): general scalars go through the plain
// kernel's operations.  With axpby_dd's one rounding chain the backward error
// of an Rtrsm of order 1300 with 150 right-hand sides was 2 % above the FP64
// pipe's in the mean square.
template <bool UPD>
__device__ __forceinline__ void crt_store(const CrtArgs &p, dd v, int64_t off, double ch, double cl) {
    dd r;
    switch (p.ab_mode) {
        case 1:   // alpha = +-1, beta = 0: the product itself
            r = p.alpha_neg ? dd{-v.hi, -v.lo} : v;
            break;
        case 2:   // alpha = +-1, beta = 1 (every Cholesky update): one dd addition
            r = add_sloppy(dd{ch, cl}, p.alpha_neg ? dd{-v.hi, -v.lo} : v);
            break;
        default:
            if (UPD && !p.beta_zero)
                r = add(p.ab_mode == 3 ? (p.alpha_neg ? dd{-v.hi, -v.lo} : v)
                                       : mul(dd{p.alpha.hi, p.alpha.lo}, v),
                        mul(dd{p.beta.hi, p.beta.lo}, dd{ch, cl}));
            else if (!p.beta_zero)
                r = axpby_dd(dd{p.alpha.hi, p.alpha.lo}, v, dd{p.beta.hi, p.beta.lo}, dd{ch, cl});
            else
                r = p.alpha_one ? v : mul(dd{p.alpha.hi, p.alpha.lo}, v);
    }
    p.ch[off] = r.hi;
    p.cl[off] = r.lo;
}

// Entry pairs (i, i + 1) of column j, i even (m_pad is even, so the pair's
// residues exist even when i + 1 = m): one 2-byte load per modulus brings both
// entries' residues, packed four moduli to a register.  (Requesting the next
// pair's loads ahead measured slower: the extra registers cost more occupancy
// than the overlap gains.)
// G: groups of four moduli, 4 (G - 1) < N <= 4 G or the weights past N zero.
template <int NW, int G, bool UPD>
__device__ __forceinline__ void crt_pair(const CrtArgs &p, const CrtTables &T, int N, int W,
                                         int64_t i, int64_t j) {
    const bool in0 = !((p.tri == 1 && i > j) || (p.tri == 2 && i < j));
    const bool in1 = i + 1 < p.m && !((p.tri == 1 && i + 1 > j) || (p.tri == 2 && i + 1 < j));
    if (!in0 && !in1) return;
    uint32_t R0[G], R1[G];
    {
        const int64_t at = j * p.m_pad + i, plane = p.n_pad * p.m_pad;
        uint32_t v[2 * G];
#pragma unroll
        for (int h = 0; h < 2 * G; ++h) {   // N is even: moduli 2h and 2h + 1
            v[h] = 0;
            if (h < 2 * (G - 1) || 2 * h < N) {
                const uint8_t *res = p.res + (int64_t)(2 * h) * plane + at;
                const uint32_t lo = __ldg(reinterpret_cast<const unsigned short *>(res));
                const uint32_t hi = __ldg(reinterpret_cast<const unsigned short *>(res + plane));
                v[h] = lo | (hi << 16);
            }
        }
#pragma unroll
        for (int g = 0; g < G; ++g) {
            R0[g] = __byte_perm(v[2 * g], v[2 * g + 1], 0x6420);   // entry i: moduli 4g .. 4g+3
            R1[g] = __byte_perm(v[2 * g], v[2 * g + 1], 0x7531);   // entry i + 1
        }
    }
    const bool use_c = p.ab_mode == 2 || (UPD && p.ab_mode == 3) ||
                       (p.ab_mode == 0 && !p.beta_zero);
    const int64_t off = i + j * p.ldc;
    const int ec = scale_exponent(__ldg(p.cmax + j)) - 2 * W;
    double c0h = 0.0, c0l = 0.0, c1h = 0.0, c1l = 0.0;
    if (use_c && in0) {
        c0h = p.ch[off];
        c0l = p.cl[off];
    }
    if (use_c && in1) {
        c1h = p.ch[off + 1];
        c1l = p.cl[off + 1];
    }
    if (in0) {
        uint32_t Z[NW];
        crt_integer<NW, G>(T, R0, Z);
        dd v;
        bigf::signed_words_to_dd<NW>(Z, scale_exponent(__ldg(p.rmax + i)) + ec, v.hi, v.lo);
        crt_store<UPD>(p, v, off, c0h, c0l);
    }
    if (in1) {
        uint32_t Z[NW];
        crt_integer<NW, G>(T, R1, Z);
        dd v;
        bigf::signed_words_to_dd<NW>(Z, scale_exponent(__ldg(p.rmax + i + 1)) + ec, v.hi, v.lo);
        crt_store<UPD>(p, v, off + 1, c1h, c1l);
    }
}

// One entry (i, j): the pair's 2-byte loads (shared with the neighbouring
// lane), the entry's bytes picked out of them.
template <int NW, int G, bool UPD>
__device__ __forceinline__ void crt_one(const CrtArgs &p, const CrtTables &T, int N, int W,
                                        int64_t i, int64_t j) {
    if ((p.tri == 1 && i > j) || (p.tri == 2 && i < j)) return;
    uint32_t R[G];
    const int64_t at = j * p.m_pad + (i & ~(int64_t)1), plane = p.n_pad * p.m_pad;
    const uint32_t sel = (i & 1) ? 0x7531u : 0x6420u;
    uint32_t v[2 * G];
#pragma unroll
    for (int h = 0; h < 2 * G; ++h) {
        v[h] = 0;
        if (h < 2 * (G - 1) || 2 * h < N) {
            const uint8_t *res = p.res + (int64_t)(2 * h) * plane + at;
            const uint32_t lo = __ldg(reinterpret_cast<const unsigned short *>(res));
            const uint32_t hi = __ldg(reinterpret_cast<const unsigned short *>(res + plane));
            v[h] = lo | (hi << 16);
        }
    }
#pragma unroll
    for (int g = 0; g < G; ++g) R[g] = __byte_perm(v[2 * g], v[2 * g + 1], sel);
    const bool use_c = p.ab_mode == 2 || (UPD && p.ab_mode == 3) ||
                       (p.ab_mode == 0 && !p.beta_zero);
    const int64_t off = i + j * p.ldc;
    const double ch = use_c ? p.ch[off] : 0.0, cl = use_c ? p.cl[off] : 0.0;
    const int sc = scale_exponent(__ldg(p.rmax + i)) + scale_exponent(__ldg(p.cmax + j)) - 2 * W;
    uint32_t Z[NW];
    crt_integer<NW, G>(T, R, Z);
    dd v2;
    bigf::signed_words_to_dd<NW>(Z, sc, v2.hi, v2.lo);
    crt_store<UPD>(p, v2, off, ch, cl);
}

template <int NW, int G, bool UPD>
__device__ __forceinline__ void crt_loop(const CrtArgs &p, const CrtTables &T, int N, int W) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p.single) {   // the grid has a thread for every entry
        const int64_t j = idx / p.m;
        if (j < p.n) crt_one<NW, G, UPD>(p, T, N, W, idx - j * p.m, j);
        return;
    }
    // pair index = j * mh + ih, kept as (ih, j); the stride likewise
    const int64_t mh = (p.m + 1) / 2;
    int64_t j = idx / mh, ih = idx - j * mh;
    const int64_t sj = stride / mh, si = stride - sj * mh;
    while (j < p.n) {
        crt_pair<NW, G, UPD>(p, T, N, W, 2 * ih, j);
        ih += si;
        j += sj;
        if (ih >= mh) {
            ih -= mh;
            ++j;
        }
    }
}

// Words and groups of four moduli of the three candidate widths for every k
// the form takes: at 112 bits 8 words and N = 30 or 32 up to k = 32768, 9 words
// and N = 34 beyond; at 120 bits 9 words and N = 34 or 36; at 128 bits 9 or 10
// words and N = 36 or 38 (more words or groups than needed give the same
// result: their weights are zero).  They are compile-time constants: with a
// test of the count in every word's loop a quarter of the instructions were
// tests and branches.
template <int NW0, int G0, bool UPD>
__global__ void __launch_bounds__(256, 4) crt_kernel(const __grid_constant__ CrtArgs p) {
    chain_begin();
    if (p.info != nullptr && *p.info != 0) return;   // an earlier step failed
    const PlanPick pk = plan_choice(p.plan);
    if (pk.c < 0) return;                            // the plain kernel computes C
    if (pk.c == 0) crt_loop<NW0, G0, UPD>(p, p.tab[0], pk.count, pk.width);
    else if (pk.c == 1) crt_loop<9, 9, UPD>(p, p.tab[1], pk.count, pk.width);
    else crt_loop<10, 10, UPD>(p, p.tab[2], pk.count, pk.width);
}

// ------------------------------------------------------------------ host

// 256-thread blocks of the two crt_kernel instantiations resident per SM
// (occupancy query, once per instantiation; 1 if the query fails).
int crt_resident_blocks(int which) {
    static int cached[2] = {0, 0};
    static std::once_flag once[2];
    std::call_once(once[which], [which] {
        int b = 0;
        const void *f = which == 0 ? (const void *)crt_kernel<8, 8, false>
                                   : (const void *)crt_kernel<9, 9, false>;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, f, 256, 0) != cudaSuccess) {
            cudaGetLastError();
            b = 0;
        }
        cached[which] = b > 0 ? b : 1;
    });
    return cached[which];
}

// Little-endian multiword helpers (host).
using Big = std::vector<uint32_t>;

Big big_mul_small(const Big &a, uint32_t s) {
    Big r(a.size() + 1, 0);
    uint64_t c = 0;
    for (size_t i = 0; i < a.size(); ++i) {
        uint64_t v = (uint64_t)a[i] * s + c;
        r[i] = (uint32_t)v;
        c = v >> 32;
    }
    r[a.size()] = (uint32_t)c;
    while (r.size() > 1 && r.back() == 0) r.pop_back();
    return r;
}

Big big_div_small(const Big &a, uint32_t s, uint32_t *rem) {
    Big r(a.size(), 0);
    uint64_t c = 0;
    for (size_t i = a.size(); i-- > 0;) {
        uint64_t v = (c << 32) | a[i];
        r[i] = (uint32_t)(v / s);
        c = v % s;
    }
    if (rem) *rem = (uint32_t)c;
    while (r.size() > 1 && r.back() == 0) r.pop_back();
    return r;
}

int big_bits(const Big &a) {
    for (size_t i = a.size(); i-- > 0;)
        if (a[i]) return (int)(32 * i + 32 - __builtin_clz(a[i]));
    return 0;
}

uint32_t inv_mod(uint32_t a, uint32_t p) {   // a^-1 mod p (gcd(a, p) = 1)
    int64_t t = 0, nt = 1, r = p, nr = a % p;
    while (nr) {
        int64_t q = r / nr, tmp = t - q * nt;
        t = nt;
        nt = tmp;
        tmp = r - q * nr;
        r = nr;
        nr = tmp;
    }
    if (t < 0) t += p;
    return (uint32_t)t;
}

// Smallest even moduli count with P >= k 2^(2W) > 4 max |A' B'| (|A'|,
// |B'| < 2^(W-1)); -1 when the 40 moduli do not reach it.
int moduli_count(int64_t k, int W) {
    static int bits[kMaxMod + 1];   // of the products of the first N moduli
    static std::once_flag once;
    std::call_once(once, [] {
        Big P{1};
        for (int N = 1; N <= kMaxMod; ++N) {
            P = big_mul_small(P, modulus(N - 1));
            bits[N] = big_bits(P);
        }
    });
    const int need = 2 * W + (int)std::ceil(std::log2((double)(k > 1 ? k : 1)));
    for (int N = 1; N <= kMaxMod; ++N)
        if (bits[N] > need) {                            // P >= 2^need
            const int even = N % 2 ? N + 1 : N;          // residues come in pairs
            return even <= kMaxMod ? even : -1;
        }
    return -1;
}

// Candidate widths of a call: 112, 120 and 128 bits, with their moduli counts.
int crt_candidates(int64_t k, int *widths, int *counts) {
    int nc = 0;
    for (int D = kMinDigits; D <= kMaxDigits; ++D) {
        const int N = moduli_count(k, 8 * D);
        if (N < 0) break;
        widths[nc] = 8 * D;
        counts[nc] = N;
        ++nc;
    }
    return nc;
}

struct CrtLayout {
    int N;                                 // moduli the workspace holds (the widest candidate)
    int64_t m_pad, n_pad, k_pad;
    size_t off_rowmax, off_colmax, off_ra, off_rb, off_res, off_ma, off_mb, total;
};

size_t align1k(size_t x) { return (x + 1023) / 1024 * 1024; }

// Tile width of the residue products: 256 (twice the flops of a 128-wide tile in
// about its time, see band_tn) once there are 128 (modulus, tile) work items
// and the wider padding of n adds at most n / 8.  Band phase on 128 / 256
// columns: 64 x 1024 x 128 (128 items) 12.0 / 10.5 us, 512^3 (256) 22.7 / 17.5,
// 768^3 49 / 33; 256^3 (64) 10.2 either way, 128 x 256 x 128 (32) 8.2 / 10.2.
int crt_band_tn(int64_t m, int64_t n, int N) {
    const int64_t items = ceil_div(imax(m, 1), kBandTM) * ceil_div(imax(n, 1), 256) * N;
    const int64_t pad256 = ceil_div(imax(n, 1), 256) * 256;
    const int64_t pad128 = ceil_div(imax(n, 1), 128) * 128;
    return (items >= 128 && (pad256 - pad128) * 8 <= imax(n, 1)) ? 256 : 128;
}

// sym: the Rsyrk form, op(B) = op(A)^T (m = n): one set of maxima and
// residue planes serves both operands, padded alike (m_pad = n_pad).
CrtLayout crt_layout(int64_t m, int64_t n, int64_t k, bool sym = false) {
    CrtLayout L{};
    int widths[kMaxCand], counts[kMaxCand];
    const int nc = crt_candidates(k, widths, counts);
    L.N = nc > 0 ? counts[nc - 1] : -1;
    const int TN = crt_band_tn(m, n, L.N);
    L.n_pad = ceil_div(imax(n, 1), TN) * TN;
    L.m_pad = sym ? L.n_pad : ceil_div(imax(m, 1), kBandTM) * kBandTM;
    L.k_pad = ceil_div(imax(k, 1), kBandTK) * kBandTK;
    const size_t N = L.N > 0 ? (size_t)L.N : 0;
    size_t o = 1024;
    L.off_rowmax = o; o = align1k(o + 8 * (size_t)L.m_pad);
    L.off_colmax = sym ? L.off_rowmax : o;
    if (!sym) o = align1k(o + 8 * (size_t)L.n_pad);
    L.off_ra = o; o = align1k(o + 2 * N * L.m_pad * L.k_pad);
    L.off_rb = sym ? L.off_ra : o;
    if (!sym) o = align1k(o + 2 * N * L.n_pad * L.k_pad);
    L.off_res = o; o = align1k(o + N * L.n_pad * L.m_pad);
    L.off_ma = o; o = align1k(o + 2 * (size_t)L.m_pad * L.k_pad);
    L.off_mb = sym ? L.off_ma : o;
    if (!sym) o = align1k(o + 2 * (size_t)L.n_pad * L.k_pad);
    L.total = o;
    return L;
}

// Residues of the call's operands (b == nullptr: one) in one launch of the
// blocks resident at once, shared out by the operands' padded rows.
int launch_residues(const SplitOperand &a, __half *ra, const SplitOperand *b, __half *rb, int64_t k,
                    int64_t k_pad, const SplitPlan &plan, cudaStream_t st) {
    ResOperand x{a.hi, a.lo, a.ld, a.row_contig, a.rows, a.rows_pad, a.max, ra, 0}, y{};
    if (b) y = ResOperand{b->hi, b->lo, b->ld, b->row_contig, b->rows, b->rows_pad, b->max, rb, 0};
    const int64_t slots = (int64_t)sm_count() * kResBlocks;
    auto items = [&](const ResOperand &o) {   // block items
        return o.row_contig ? o.rows_pad / 16 * (k_pad / 64)
                            : ceil_div(o.rows_pad * (k_pad / 64), kResWarps);
    };
    // a block item takes its warps two rows (row-contiguous) or one
    const int64_t ia = items(x), ib = items(y), ca = x.row_contig ? 2 : 1, cb = y.row_contig ? 2 : 1;
    int64_t na = ia, nb = ib;
    if (ia + ib > slots) {
        na = slots * (ia * ca) / (ia * ca + ib * cb);
        na = na < 1 ? 1 : na > ia ? ia : na;
        nb = slots - na < ib ? slots - na : ib;
        if (b && nb < 1) nb = 1;
        // few rounds: the split with the shortest longest one
        if (b && ia * ca + ib * cb <= 16 * slots) {
            int64_t best = -1;
            for (int64_t r = 1; r <= 16; ++r) {
                const int64_t ta = ceil_div(ia, r), tb = slots - ta;
                if (tb < 1) continue;
                const int64_t q = ceil_div(ib, tb), t = r * ca > q * cb ? r * ca : q * cb;
                if (best < 0 || t < best) {
                    best = t;
                    na = ta;
                    nb = ceil_div(ib, q);
                }
            }
        }
    }
    x.blocks = (unsigned)na;
    y.blocks = (unsigned)nb;
    return chained_ok(launch_chained_if(ia + ib <= 4 * slots, residue_kernel, (unsigned)(na + nb),
                                        kResThreads, 0, st, x, y, k, k_pad, plan),
                      "residue_kernel");
}

// Reconstruction constants for the first N moduli, formed with multiword
// integers on the host.
int make_crt_tables(int N, CrtTables &T, int *nwords) {
    memset(&T, 0, sizeof T);
    Big P{1};
    for (int i = 0; i < N; ++i) P = big_mul_small(P, modulus(i));
    if ((int)P.size() > kWords - 1) return fail(MP_DD_ERR_TOO_LARGE, "moduli product too wide");
    {   // 2^(32 kWords) - P
        uint64_t borrow = 0;
        for (int t = 0; t < kWords; ++t) {
            const uint64_t d = 0 - (uint64_t)(t < (int)P.size() ? P[t] : 0u) - borrow;
            T.negp[2 * t] = (uint32_t)d & 0xFFFFu;
            T.negp[2 * t + 1] = ((uint32_t)d >> 16) & 0xFFFFu;
            borrow = (d >> 63) & 1;
        }
    }
    for (int i = 0; i < N; ++i) {
        uint32_t mi_mod = 0;
        Big Mi = big_div_small(P, modulus(i), nullptr);
        big_div_small(Mi, modulus(i), &mi_mod);
        const uint32_t inv = inv_mod(mi_mod, modulus(i));
        Big wi = big_mul_small(Mi, inv);
        const int g = i / 4, sh = 8 * (i % 4);
        for (int t = 0; t < 4 * kWords; ++t) {
            const uint32_t word = t / 4 < (int)wi.size() ? wi[t / 4] : 0u;
            T.wp[g][t] |= ((word >> (8 * (t % 4))) & 0xFFu) << sh;
        }
        const uint32_t qfix = (uint32_t)((((uint64_t)inv << 24) + modulus(i) / 2) / modulus(i));
        for (int t = 0; t < 3; ++t) T.qp[g][t] |= ((qfix >> (8 * t)) & 0xFFu) << sh;
    }
    // words of the sums: S = sum_b c_b w_b < N 255 P, and Z = S - q P takes
    // a sign bit: bits(P) + ceil(log2(255 N)) + 1
    int need = big_bits(P) + 1;
    for (int64_t x = 255LL * N - 1; x > 0; x >>= 1) ++need;
    *nwords = (need + 31) / 32;
    return 0;
}

// The same, formed once per N and process (forming them took ~8 us per
// candidate width and call: 56 us of host time per call, 32 since).
int crt_tables(int N, CrtTables &T, int *nwords) {
    struct Entry {
        std::once_flag once;
        CrtTables T;
        int words = 0, rc = 0;
    };
    static Entry cache[kMaxMod + 1];
    if (N < 1 || N > kMaxMod) return fail(MP_DD_ERR_TOO_LARGE, "%d moduli", N);
    Entry &e = cache[N];
    std::call_once(e.once, [&] { e.rc = make_crt_tables(N, e.T, &e.words); });
    if (e.rc) return fail(e.rc, "moduli product too wide");
    T = e.T;
    *nwords = e.words;
    return 0;
}

}  // namespace

size_t crt_workspace_bytes(int64_t m, int64_t n, int64_t k, bool sym) {
    return crt_layout(m, n, k, sym).total;
}

double crt_estimate_us(int64_t m, int64_t n, int64_t k) {
    // launches and latencies, then reconstruction, residues and products; fitted
    // to 64 x 2048 x 192 66 us, 512^3 80, 1024^3 181, 1501 x 2777 x 1999 757, before
    // the small kernels of a call were shortened (512^3: 58 us), so that products
    // near the rule's line stay on the FP64 pipe a little longer than they need
    const double dm = (double)m, dn = (double)n, dk = (double)k;
    return 60.0 + 4e-5 * dm * dn + 1.6e-5 * (dm + dn) * dk + 5e-8 * dm * dn * dk;
}

int crt_layout_query(int64_t m, int64_t n, int64_t k, size_t *off, int *count) {
    CrtLayout L = crt_layout(m, n, k);
    off[0] = L.off_rowmax;
    off[1] = L.off_colmax;
    off[2] = L.off_ra;
    off[3] = L.off_rb;
    off[4] = L.off_res;
    off[5] = (size_t)L.m_pad;
    off[6] = (size_t)L.n_pad;
    off[7] = (size_t)L.k_pad;
    *count = L.N;
    for (int i = 0; i < L.N && i < kMaxMod; ++i) off[8 + i] = (size_t)modulus(i);
    return 0;
}

int crt_magnitude_offsets(int64_t m, int64_t n, int64_t k, bool sym, size_t *off) {
    CrtLayout L = crt_layout(m, n, k, sym);
    off[0] = L.off_ma;
    off[1] = L.off_mb;
    return 0;
}

int run_crt(const GemmArgs &p, void *ws, size_t ws_bytes, cudaStream_t st) {
    if (p.k > ((int64_t)1 << 17) - 1)
        return fail(MP_DD_ERR_TOO_LARGE, "k = %lld exceeds 131071 (int32 products)",
                    (long long)p.k);
    // the Rsyrk form: one triangle of op(A) op(A)^T
    const bool sym = p.tri != 0;
    if (sym && (p.m != p.n || p.ah != p.bh || p.al != p.bl || p.lda != p.ldb || p.ta == p.tb))
        return fail(MP_DD_ERR_TOO_LARGE, "CRT Rsyrk: operands are not A and A^T");
    CrtLayout L = crt_layout(p.m, p.n, p.k, sym);
    int widths[kMaxCand], counts[kMaxCand];
    const int ncand = crt_candidates(p.k, widths, counts);
    if (ncand < 1 || L.N < 0 || L.N > kMaxMod)
        return fail(MP_DD_ERR_TOO_LARGE, "k too large for the moduli");
    if (ws == nullptr || ws_bytes < L.total)
        return fail(MP_DD_ERR_WORKSPACE, "CRT Rgemm needs %zu workspace bytes, got %zu",
                    L.total, ws_bytes);
    if ((int64_t)L.N * L.m_pad > 0x7fffffffLL || (int64_t)L.N * L.n_pad > 0x7fffffffLL)
        return fail(MP_DD_ERR_TOO_LARGE, "matrix too large for the CRT path");
    const int TN = crt_band_tn(p.m, p.n, L.N);

    uint8_t *w = static_cast<uint8_t *>(ws);
    cudaError_t e = cudaMemsetAsync(w, 0, L.off_ra, st);   // header (form 0) and maxima
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemsetAsync");
    if (p.alpha_zero) return launch_gemm_plain(p, st);
    auto *rmax = reinterpret_cast<unsigned long long *>(w + L.off_rowmax);
    auto *cmax = reinterpret_cast<unsigned long long *>(w + L.off_colmax);
    auto *RA = reinterpret_cast<__half *>(w + L.off_ra);
    auto *RB = reinterpret_cast<__half *>(w + L.off_rb);
    auto *RES = reinterpret_cast<uint8_t *>(w + L.off_res);
    auto *hdr = reinterpret_cast<SplitHeader *>(w);

    double cst[kMaxCand];
    for (int c = 0; c < ncand; ++c) cst[c] = 1.0 + 0x1p-50;   // (1 + 2^-W), rounded up
    if (p.tight > 0.0)   // thresholds for tight u^2 instead of 12 k u^2
        for (int c = 0; c < ncand; ++c) cst[c] *= 12.0 * (double)p.k / p.tight;
    SplitHeader init;
    const SplitPlan plan = make_plan(&init, &hdr->dmin, 2, p.k, ncand, widths, counts, cst);

    const int a_rc = p.ta ? 0 : 1, b_rc = p.tb ? 1 : 0;
    int rc;
    // (an update inside a solve or factorisation is not one of the timed calls)
    auto mark = [&](int phase) {
        if (p.tight == 0.0) sliced_timing_mark(phase, st);
    };
    mark(0);
    const SplitOperand oa{p.ah, p.al, p.lda, a_rc, p.m, L.m_pad, rmax, w + L.off_ma, 0};
    const SplitOperand ob{p.bh, p.bl, p.ldb, b_rc, p.n, L.n_pad, cmax, w + L.off_mb, 0};
    // (the Rsyrk form has one operand: its maxima and planes serve as both)
    if ((rc = launch_absmax(oa, sym ? nullptr : &ob, p.k, st))) return rc;
    if ((rc = launch_magnitude(oa, sym ? nullptr : &ob, p.k, L.k_pad, hdr, init, st))) return rc;
    if ((rc = launch_certificate(p, w + L.off_ma, w + L.off_mb, L.m_pad, L.n_pad, L.k_pad, TN,
                                 rmax, cmax, hdr, st)))
        return rc;
    if ((rc = launch_residues(oa, RA, sym ? nullptr : &ob, RB, p.k, L.k_pad, plan, st))) return rc;

    mark(1);
    CUtensorMap tmA, tmB;
    if ((rc = make_tmap(&tmA, RA, (int64_t)L.N * L.m_pad, L.k_pad, kBandTM))) return rc;
    if ((rc = make_tmap(&tmB, RB, (int64_t)L.N * L.n_pad, L.k_pad, TN))) return rc;
    CUtensorMap tmB_half;   // half-height boxes for CTA pairs on 256-wide tiles
    if ((rc = make_tmap(&tmB_half, RB, (int64_t)L.N * L.n_pad, L.k_pad, TN / 2))) return rc;
    BandArgs ba{};
    ba.S = L.N;
    ba.kb_count = (int)(L.k_pad / kBandTK);
    ba.tiles_m = (int)(L.m_pad / kBandTM);
    ba.tiles_n = (int)(L.n_pad / TN);
    ba.m_pad = L.m_pad;
    ba.n_pad = L.n_pad;
    ba.P = nullptr;
    ba.R = RES;
    ba.hdr = hdr;
    ba.diag = 1;
    ba.tri = p.tri;
    ba.plan = plan;
    for (int i = 0; i < L.N; ++i) {
        const int p_i = modulus(i), r = p_i / 2;   // residues: |r| <= 128 mod 256, (p - 1) / 2
        ba.moduli[i] = p_i;
        ba.run_kb[i] = (1 << 24) / (r * r) / kBandTK;   // r^2 64 run_kb <= 2^24
    }
    if ((rc = launch_band(tmA, tmB, ba, TN, st, &tmB_half))) return rc;
    mark(2);

    // CRT constants of every candidate
    CrtArgs ca{};
    ca.plan = plan;
    ca.m = p.m; ca.n = p.n; ca.m_pad = L.m_pad; ca.n_pad = L.n_pad;
    ca.res = RES; ca.rmax = rmax; ca.cmax = sym ? rmax : cmax;
    ca.alpha = p.alpha; ca.beta = p.beta;
    ca.alpha_one = p.alpha_one; ca.beta_zero = p.beta_zero;
    ca.ch = p.ch; ca.cl = p.cl; ca.ldc = p.ldc;
    ca.tri = p.tri;
    ca.info = p.info;
    {
        const bool a_pm1 = p.alpha.lo == 0.0 && (p.alpha.hi == 1.0 || p.alpha.hi == -1.0);
        const bool b_one = p.beta.hi == 1.0 && p.beta.lo == 0.0;
        ca.ab_mode = !a_pm1 ? 0 : p.beta_zero ? 1 : b_one ? 2 : p.tight > 0.0 ? 3 : 0;
        ca.alpha_neg = p.alpha.hi < 0.0;
    }
    int nw[kMaxCand] = {0, 0, 0};
    for (int c = 0; c < ncand; ++c)
        if ((rc = crt_tables(counts[c], ca.tab[c], &nw[c]))) return rc;
    const int which = nw[0] <= 8 && counts[0] <= 32 ? 0 : 1;
    const int words[kMaxCand] = {which == 0 ? 8 : 9, 9, 10};
    for (int c = 0; c < ncand; ++c)   // (see crt_kernel)
        if (nw[c] > words[c] || counts[c] > 4 * words[c] || counts[c] < 4 * words[c] - 4)
            return fail(MP_DD_ERR_TOO_LARGE, "CRT words %d / moduli %d beyond the kernel's", nw[c],
                        counts[c]);
    // one thread per entry pair, looping.  Full products: as many blocks as
    // are resident at once (four per SM; eight per SM left
    // the last two-thirds wave with a third of the slots idle: 3.65-3.68
    // against 3.70-3.73 ms at 8192).  Triangles: eight per SM, which the
    // block scheduler balances over the uneven work of the skipped entries
    // (resident blocks only: 2.61 against 2.41-2.45 ms).
    const int64_t pairs = ceil_div(p.m, 2) * p.n;
    int64_t blocks = ceil_div(pairs, 256);
    const int64_t cap = (int64_t)sm_count() * (p.tri ? 8 : crt_resident_blocks(which));
    // few entries: one per thread halves the latency of a thread's chain (64 x
    // 2048: 17.3 us in pairs, 15.4 so; 512 x 512, already two blocks per SM
    // and more: 21.4 either way)
    ca.single = p.m * p.n <= 2 * 256 * (int64_t)sm_count() * crt_resident_blocks(which);
    if (ca.single) blocks = ceil_div(p.m * p.n, 256);
    else if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    const unsigned nb = (unsigned)blocks;
    void (*const kernel)(CrtArgs) =
        p.tight > 0.0 ? (which == 0 ? crt_kernel<8, 8, true> : crt_kernel<9, 9, true>)
                      : (which == 0 ? crt_kernel<8, 8, false> : crt_kernel<9, 9, false>);
    const cudaError_t le = launch_chained(kernel, nb, 256, 0, st, ca);
    if ((rc = chained_ok(le, "crt_kernel"))) return rc;
    rc = launch_plain_fallback(p, plan, st);
    mark(3);
    return rc;
}

}  // namespace mpdd
