// Plain double-double Rgemm / Rsyrk kernel for sm_103a (FP64 DFMA path).
//
// Computes C := alpha op(A) op(B) + beta C (Rgemm), one triangle of
// alpha A A^T + beta C (Rsyrk) or of alpha (A B^T + B A^T) + beta C (Rsyr2k:
// the second product continues the same k loop), and alpha S B + beta C or
// alpha B S + beta C with S symmetric and one triangle stored (Rsymm: the
// operand is read through the stored triangle); MPBLAS semantics (manual
// Sec. 7.3 and the routine table of Sec. 6).  Every multiply-add is dd
// arithmetic: the exact product of the hi parts by FMA, the two cross
// products, TwoSum into the accumulator, and a TwoSum renormalisation
// every 4 steps of k (dd_arith.cuh).
//
// On GB300 the FP64 pipe is the bottleneck by a wide margin (6.25 FP64
// instructions per dd multiply-add), so the kernel is organised to keep that
// pipe busy and nothing else: each CTA owns a 16 x 16 tile of C, one dd
// accumulator per thread (a 16 x 8 or 32 x 4 tile for products that leave SMs
// without a 16 x 16 tile: four warps, one per partition of the SM, so a step of
// k takes half as long; 64 x 64 tiles of 4 x 4 accumulators a thread for
// launches behind a certificate, which mostly return at once and cost their
// CTA count, where the TMA-staged form of this kernel, dd_gemm_tma.cu, whose
// per-entry arithmetic is identical, does not apply), and the hi/lo planes
// of the op(A) and op(B) panels are staged through shared memory 16 columns
// of k at a time with a register prefetch of the next panel.  One SM's FP64
// pipe issues only 2 lanes per clock, so one chain a warp keeps it busy.
// Loads are zero-filled outside the matrices; a zero product leaves
// a normalised accumulator bitwise unchanged, so the per-entry operation
// sequence (l = 0, 1, ..., k-1) and hence the result are independent of the
// tiling.  Rsyrk uses the same instantiation as Rgemm(N, T) / (T, N) over
// the tiles of one triangle, so its entries equal Rgemm's bit for bit.
#include "common.cuh"
#include "dd_arith.cuh"
#include "kernels.cuh"
#include "ozaki_common.cuh"

namespace mpdd {
namespace {

constexpr int BK = 16;

// Tile shapes: TX x TY threads, each an R x R block of entries TX (TY) apart.
// ALONE: for launches of at most one tile per SM, whose time is the latency of
// a warp's chain, where the integer forms of the errors do not help (96 x 80 x
// 70: 31.9 us, 32.7 with the sums' on the integer pipe).
template <int R_, int TX_, int TY_, bool ALONE_ = false>
struct PlainShape {
    static constexpr bool ALONE = ALONE_;
    static constexpr int R = R_, TX = TX_, TY = TY_, NT = TX_ * TY_;
    static constexpr int BM = TX_ * R_, BN = TY_ * R_;
    static constexpr int QA = (BM * BK + NT - 1) / NT, QB = (BN * BK + NT - 1) / NT;
};
template <int R>
using Square = PlainShape<R, 16, 16>;
using Half = PlainShape<1, 16, 8>;    // 16 x 8
using Tall = PlainShape<1, 32, 4>;    // 32 x 4
using HalfAlone = PlainShape<1, 16, 8, true>;
using TallAlone = PlainShape<1, 32, 4, true>;

template <class S>
struct PlainSmem {
    double ah[BK][S::BM + 1], al[BK][S::BM + 1];  // op(A) panel, [l][i]
    double bh[BK][S::BN + 1], bl[BK][S::BN + 1];  // op(B) panel, [l][j]
};

constexpr int GROUP_N = 8;  // tile columns per rasterisation group

// Tile (bi, bj) of this CTA.  Rgemm: a 1-D grid walked in groups of GROUP_N
// tile columns with the tile row fastest inside a group, so the CTAs
// resident at one time share a few A row panels and B column panels in L2
// (a plain column-by-column order re-reads all of A for every tile column).
// Rsyrk: a 1-D grid over the square tiles of one triangle, t -> (row, col)
// with row <= col (upper) or row >= col (lower); a 16 x 8 tile is half of one.
template <int BM, int BN>
__device__ __forceinline__ void tile_coords(const GemmArgs &p, int64_t &bi, int64_t &bj) {
    if (p.tri == 0) {
        const int64_t tm = (p.m + BM - 1) / BM, tn = (p.n + BN - 1) / BN;
        const int64_t t = blockIdx.x;
        const int64_t group = t / (tm * GROUP_N);
        const int64_t first = group * GROUP_N;
        const int64_t gn = tn - first < GROUP_N ? tn - first : GROUP_N;
        const int64_t local = t - group * tm * GROUP_N;
        bj = first + local % gn;
        bi = local / gn;
        return;
    }
    constexpr int64_t kParts = BM / BN;
    int64_t t = blockIdx.x / kParts;
    int64_t r = (int64_t)((__dsqrt_rn(8.0 * (double)t + 1.0) - 1.0) * 0.5);
    while (r * (r + 1) / 2 > t) --r;
    while ((r + 1) * (r + 2) / 2 <= t) ++r;
    int64_t c = t - r * (r + 1) / 2;  // 0 <= c <= r
    if (p.tri == 1) {
        bi = c;
        bj = r;
    } else {
        bi = r;
        bj = c;
    }
    bj = bj * kParts + blockIdx.x % kParts;
}

template <int TA, int TB, class S>
__device__ __forceinline__ void plain_body(const GemmArgs &p, PlainSmem<S> &s) {
    constexpr int R = S::R, BM = S::BM, BN = S::BN, NT = S::NT, QA = S::QA, QB = S::QB;
    constexpr int TX = S::TX, TY = S::TY;
    chain_begin();
    if (p.info != nullptr && *p.info != 0) return;  // an earlier step failed
    // behind a split-precision call: compute only when its certificate failed
    if (p.gate != nullptr &&
        *reinterpret_cast<const volatile unsigned int *>(p.gate) >= p.gate_below)
        return;
    int64_t bi, bj;
    tile_coords<BM, BN>(p, bi, bj);
    const int t = threadIdx.x, tx = t % TX, ty = t / TX;
    const int64_t i0 = bi * BM, j0 = bj * BN;
    // the k loop: [0, k) over (A, B), then for Rsyr2k [k1, k1 + k) over
    // (A2, B2), k1 = k rounded up to whole panels (zero products between)
    const int64_t k1 = (p.k + BK - 1) / BK * BK;
    const int64_t kk = p.alpha_zero ? 0 : (p.a2h != nullptr ? k1 + p.k : p.k);

    dd acc[R][R];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < R; ++c) acc[r][c] = dd{0.0, 0.0};

    // a panel holds BM x 16 entries of op(A) and BN x 16 of op(B)
    double rah[QA], ral[QA], rbh[QB], rbl[QB];
    // Element q of this thread's share of a panel: (row-in-panel, l).
    auto a_pos = [&](int q, int &ii, int &ll) {
        int idx = t + NT * q;
        if (!TA) { ii = idx % BM; ll = idx / BM; }   // contiguous in i
        else     { ll = idx % BK; ii = idx / BK; }   // contiguous in l
    };
    auto b_pos = [&](int q, int &jj, int &ll) {
        int idx = t + NT * q;
        if (!TB) { ll = idx % BK; jj = idx / BK; }   // contiguous in l
        else     { jj = idx % BN; ll = idx / BN; }   // contiguous in j
    };
    auto load = [&](int64_t l0) {
        const bool second = p.a2h != nullptr && l0 >= k1;
        const double *Ah = second ? p.a2h : p.ah, *Al = second ? p.a2l : p.al;
        const double *Bh = second ? p.b2h : p.bh, *Bl = second ? p.b2l : p.bl;
        const int64_t lda = second ? p.lda2 : p.lda, ldb = second ? p.ldb2 : p.ldb;
        const int64_t lb = second ? l0 - k1 : l0;
#pragma unroll
        for (int q = 0; q < QA; ++q) {
            int ii, ll;
            a_pos(q, ii, ll);
            int64_t gi = i0 + ii, gl = lb + ll;
            bool ok = gi < p.m && gl < p.k;
            int64_t off = TA ? (gl + gi * lda) : (gi + gl * lda);
            if (p.sym_a) {
                const bool direct = p.sym_a == 1 ? gi <= gl : gi >= gl;
                off = direct ? gi + gl * lda : gl + gi * lda;
            }
            rah[q] = ok ? Ah[off] : 0.0;
            ral[q] = ok ? Al[off] : 0.0;
        }
#pragma unroll
        for (int q = 0; q < QB; ++q) {
            int jj, ll;
            b_pos(q, jj, ll);
            int64_t gj = j0 + jj, gl = lb + ll;
            bool ok = gj < p.n && gl < p.k && (BN * BK >= NT || t < BN * BK);
            int64_t off = TB ? (gj + gl * ldb) : (gl + gj * ldb);
            if (p.sym_b) {
                const bool direct = p.sym_b == 1 ? gl <= gj : gl >= gj;
                off = direct ? gl + gj * ldb : gj + gl * ldb;
            }
            rbh[q] = ok ? Bh[off] : 0.0;
            rbl[q] = ok ? Bl[off] : 0.0;
        }
    };
    auto stage = [&]() {
#pragma unroll
        for (int q = 0; q < QA; ++q) {
            int ii, ll;
            a_pos(q, ii, ll);
            s.ah[ll][ii] = rah[q];
            s.al[ll][ii] = ral[q];
        }
#pragma unroll
        for (int q = 0; q < QB; ++q) {
            int jj, ll;
            b_pos(q, jj, ll);
            if (BN * BK >= NT || t < BN * BK) {
                s.bh[ll][jj] = rbh[q];
                s.bl[ll][jj] = rbl[q];
            }
        }
    };

    if (kk > 0) {
        load(0);
        for (int64_t l0 = 0; l0 < kk; l0 += BK) {
            __syncthreads();
            stage();
            __syncthreads();
            if (l0 + BK < kk) load(l0 + BK);
#pragma unroll 1
            for (int l4 = 0; l4 < BK; l4 += kRenormEvery) {
#pragma unroll (R * R >= 8 ? 1 : kRenormEvery)
                for (int l = l4; l < l4 + kRenormEvery; ++l) {
                    dd a[R], b[R];
#pragma unroll
                    for (int r = 0; r < R; ++r)
                        a[r] = dd{s.ah[l][tx + TX * r], s.al[l][tx + TX * r]};
#pragma unroll
                    for (int c = 0; c < R; ++c)
                        b[c] = dd{s.bh[l][ty + TY * c], s.bl[l][ty + TY * c]};
#pragma unroll
                    for (int r = 0; r < R; ++r)
#pragma unroll
                        for (int c = 0; c < R; ++c) {
                            if constexpr (S::ALONE) mac_deferred(acc[r][c], a[r], b[c]);
                            else mac_mixed(acc[r][c], a[r], b[c]);
                        }
                }
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int c = 0; c < R; ++c) {
                        if constexpr (S::ALONE) renorm_exact(acc[r][c]);
                        else renorm_mixed(acc[r][c]);
                    }
            }
        }
    }

    const dd alpha{p.alpha.hi, p.alpha.lo}, beta{p.beta.hi, p.beta.lo};
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < R; ++c) {
            int64_t i = i0 + tx + TX * r, j = j0 + ty + TY * c;
            if (i >= p.m || j >= p.n) continue;
            if ((p.tri == 1 && i > j) || (p.tri == 2 && i < j)) continue;
            dd v = p.alpha_one ? acc[r][c] : mul(alpha, acc[r][c]);
            int64_t off = i + j * p.ldc;
            if (!p.beta_zero) v = add(v, mul(beta, dd{p.ch[off], p.cl[off]}));
            p.ch[off] = v.hi;
            p.cl[off] = v.lo;
        }
}

// 64 x 64 tiles (one CTA per SM by registers) and the smaller tiles (two or
// more CTAs per SM, registers capped accordingly).
template <int TA, int TB>
__global__ void __launch_bounds__(256) dd_gemm_plain_kernel(const GemmArgs p) {
    __shared__ PlainSmem<Square<4>> s;
    plain_body<TA, TB, Square<4>>(p, s);
}

template <int TA, int TB, class S>
__global__ void __launch_bounds__(S::NT, 2) dd_gemm_plain_small_kernel(const GemmArgs p) {
    __shared__ PlainSmem<S> s;
    plain_body<TA, TB, S>(p, s);
}

}  // namespace

namespace {

int64_t tile_count(const GemmArgs &p, int bm, int bn) {
    const int64_t tm = ceil_div(p.m, bm);
    return p.tri == 0 ? tm * ceil_div(p.n, bn) : tm * (tm + 1) / 2 * (bm / bn);
}

template <int TA, int TB, class S>
void launch_one(dim3 grid, const GemmArgs &p, cudaStream_t stream) {
    if constexpr (S::R == 4)
        launch_chained(dd_gemm_plain_kernel<TA, TB>, grid, S::NT, 0, stream, p);
    else
        launch_chained(dd_gemm_plain_small_kernel<TA, TB, S>, grid, S::NT, 0, stream, p);
}

template <class S>
int launch_shape(const GemmArgs &p, cudaStream_t stream) {
    const int64_t tiles = tile_count(p, S::BM, S::BN);
    if (tiles > 0x7fffffffLL) return fail(MP_DD_ERR_TOO_LARGE, "m x n too large");
    const dim3 grid((unsigned)tiles);
    if (p.ta == 0 && p.tb == 0) launch_one<0, 0, S>(grid, p, stream);
    else if (p.ta == 1 && p.tb == 0) launch_one<1, 0, S>(grid, p, stream);
    else if (p.ta == 0 && p.tb == 1) launch_one<0, 1, S>(grid, p, stream);
    else launch_one<1, 1, S>(grid, p, stream);
    return check_launch("dd_gemm_plain_kernel");
}

}  // namespace

// Tile size: the time of a launch is about (tiles per SM, rounded up) x
// (work per tile), in units of 128 entries -- one accumulator for each of four
// warps, one per partition of the SM, 0.23 us per step of k (6.25 FP64
// instructions per multiply-add at 526 G/s over 152 SMs); the per-entry
// operation sequence, and hence the result, does not depend on the tile.
// 16 x 16 tiles never take longer by that count than larger ones, and their
// six or more warps a partition hide the multiply-add's long integer part best: 8192
// x 8192 x 256 takes 197.2 ms on them, 198.1 on 32 x 32 tiles, 212 on 64 x 64
// and 222 on the TMA-staged 64 x 64 (two warps a partition); 1216 x 1024 x 512
// 7.28, 7.33, 7.86 and 8.27 ms.  16 x 8 and 32 x 4 tiles are one unit: they
// halve the time of products with fewer 16 x 16 tiles than SMs, and of those
// with few columns, whose 16-column tiles are mostly padding: Rgemm 96 x 80 x
// 70 58.0 -> 31.9 us; Cholesky and solve of order 3000, whose updates have a
// depth of 64, 36.5 -> 33.2 ms.
int64_t plain_tile_cost(const GemmArgs &p, int r) {
    const int64_t sms = sm_count() > 0 ? sm_count() : 152;
    return ceil_div(tile_count(p, 16 * r, 16 * r), sms) * 2 * r * r;
}

namespace {

enum PlainTile { kTile16, kTileHalf, kTileTall };

PlainTile plain_tile(const GemmArgs &p, int64_t *cost) {
    const int64_t sms = sm_count() > 0 ? sm_count() : 152;
    PlainTile best = kTile16;
    *cost = plain_tile_cost(p, 1);
    auto offer = [&](PlainTile t, int64_t c) {
        if (c < *cost) {
            *cost = c;
            best = t;
        }
    };
    offer(kTileHalf, ceil_div(tile_count(p, Half::BM, Half::BN), sms));
    if (p.tri == 0) offer(kTileTall, ceil_div(tile_count(p, Tall::BM, Tall::BN), sms));
    return best;
}

}  // namespace

int64_t plain_best_cost(const GemmArgs &p) {
    int64_t cost;
    plain_tile(p, &cost);
    return cost;
}

// The plain kernel behind a split-precision call: the same launch, gated on
// the call's certificate (every CTA returns at once when a width certified
// the bound).
int launch_plain_fallback(const GemmArgs &p, const SplitPlan &plan, cudaStream_t stream) {
    GemmArgs q = p;
    q.gate = plan.dmin;
    q.gate_below = plan.thr[plan.ncand - 1];
    // with the gate closed every CTA returns at once, so the launch costs
    // about its CTA count: 64 x 64 tiles, TMA-staged where that applies, else
    // register-staged whenever they fill the SMs twice (the result does not
    // depend on the staging or the tile size)
    int rc = 0;
    if (try_launch_gemm_tma(q, stream, &rc)) return rc;
    const int64_t sms = sm_count() > 0 ? sm_count() : 152;
    if (tile_count(q, 64, 64) >= 2 * sms) return launch_shape<Square<4>>(q, stream);
    return launch_gemm_plain(q, stream);
}

// Where the residue form takes an update of a factorisation or solve over
// from the plain kernel: where its estimated time is at most four fifths of
// the plain kernel's busiest SM's (plain_tile_cost).  LU and solve of order 1536
// with 500 right-hand sides: 71.0 ms with every update on the FP64 pipe
// (9.75 instructions a multiply-add), 31.9 so.
// The inner dimension and both outer ones have to reach kUpdateMin: below it
// the time is latency either way, and so solves of up to 95 right-hand sides
// never leave the FP64 pipe and each one's result is its own.  From there on the
// estimates depend on the number of columns, and the operand width on all of
// their values, so a right-hand side's low bits can differ with the others that
// go with it (within the bound of either form).
// With `tight` = 2 the residue form's operand rounding stays within 2 u^2
// (|A||B| + |C|) entry by entry, and its other roundings within 4 u^2, against
// the plain kernel's sum of k roundings of up to ~8 u^2; a call whose operands
// do not allow that at 128 bits, or hold an infinity or NaN, is computed by
// the plain kernel behind it.
constexpr int64_t kUpdateMin = 96;
constexpr double kTightUpdate = 2.0;
constexpr size_t kUpdateScratch = size_t(4) << 30;   // larger updates go in blocks

int launch_gemm_update(const GemmArgs &p, cudaStream_t stream) {
    if (p.m < kUpdateMin || p.n < kUpdateMin || p.k < kUpdateMin || p.k > ((int64_t)1 << 17) - 1 ||
        p.tri != 0 || p.alpha_zero || p.a2h != nullptr || p.sym_a || p.sym_b)
        return launch_gemm_plain(p, stream);
    const double plain_us = 0.23 * (double)p.k * (double)plain_best_cost(p);
    if (crt_estimate_us(p.m, p.n, p.k) > 0.8 * plain_us) return launch_gemm_plain(p, stream);
    // allocations inside a stream capture would belong to the graph
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return launch_gemm_plain(p, stream);
    }
    int64_t bm = p.m, bn = p.n;
    while (crt_workspace_bytes(bm, bn, p.k) > kUpdateScratch) {
        int64_t &big = bm > bn ? bm : bn;
        if (big <= 1024) return launch_gemm_plain(p, stream);
        big = ceil_div(big / 2, (int64_t)256) * 256;
    }
    const size_t bytes = crt_workspace_bytes(bm, bn, p.k);
    void *ws = nullptr;
    if (pool_alloc(&ws, bytes, stream, kPoolScratch) != cudaSuccess) {
        cudaGetLastError();
        return launch_gemm_plain(p, stream);
    }
    int rc = 0;
    for (int64_t j = 0; j < p.n && rc == 0; j += bn)
        for (int64_t i = 0; i < p.m && rc == 0; i += bm) {
            GemmArgs q = p;
            q.m = p.m - i < bm ? p.m - i : bm;
            q.n = p.n - j < bn ? p.n - j : bn;
            const int64_t oa = p.ta ? i * p.lda : i, ob = p.tb ? j : j * p.ldb;
            q.ah += oa; q.al += oa;
            q.bh += ob; q.bl += ob;
            q.ch += i + j * p.ldc; q.cl += i + j * p.ldc;
            q.tight = kTightUpdate;
            rc = run_crt(q, ws, bytes, stream);
        }
    const cudaError_t e = cudaFreeAsync(ws, stream);
    if (rc == 0 && e != cudaSuccess) return cuda_fail(e, "update workspace");
    return rc;
}

int launch_gemm_plain(const GemmArgs &p, cudaStream_t stream) {
    int rc = 0;
    if (try_launch_gemm_tma(p, stream, &rc)) return rc;
    int64_t cost;
    const PlainTile t = plain_tile(p, &cost);
    switch (t) {   // cost 1: one small tile per SM at most
        case kTileTall:
            return cost <= 1 ? launch_shape<TallAlone>(p, stream) : launch_shape<Tall>(p, stream);
        case kTileHalf:
            return cost <= 1 ? launch_shape<HalfAlone>(p, stream) : launch_shape<Half>(p, stream);
        default: return launch_shape<Square<1>>(p, stream);
    }
}

}  // namespace mpdd
