"""dd Rtrsm through the C ABI (GPU).

Pins: every side/uplo/trans/diag variant recovers an exact integer solution
bit for bit (the unused triangle, padding rows and a unit diagonal hold NaN,
so a stray read shows); ragged sizes that span several 64-row blocks and
both recursion orders meet the componentwise backward-error bound with the
residual evaluated by the oracle's exact tier, and agree with the oracle's
substitution within the forward error that the bound allows on these
diagonally dominant matrices; the ill-conditioned Cholesky factor of a
served request meets the same backward bound; alpha = 0, empty sizes and
illegal arguments behave as DTRSM; repeated calls are bitwise identical.
"""
from __future__ import annotations

import numpy as np
import pytest
import torch

import datagen
import oracle
from gpucase import dev, host
from trsmcheck import TRSM_VARIANTS, op_triangle, trsm_residual_over_bound

pytestmark = pytest.mark.gpu


def gpu_trsm(mp, c):
    A, B = dev(c.A), dev(c.B)
    mp.mp_dd_Rtrsm(c.side, c.uplo, c.transa, c.diag, c.m, c.n, c.alpha, A, c.A[0].shape[0], B,
                   c.B[0].shape[0])
    return host(B, c.m, c.n)


def integer_case(side, uplo, transa, diag, m, n, seed):
    """A TrsmCase whose solution is the integer matrix X: A has small integer
    entries and a power-of-two diagonal, alpha = 2 and B = op(A) X / 2 (or
    X op(A) / 2), exact in binary64."""
    g = datagen.rng(seed)
    order = m if side == "L" else n
    A = g.integers(-3, 4, (order, order)).astype(np.float64)
    np.fill_diagonal(A, g.choice([-2.0, -1.0, 1.0, 2.0], order))
    X = g.integers(-9, 10, (m, n)).astype(np.float64)
    T = op_triangle(A, uplo, transa, diag, order)
    Bx = (T @ X if side == "L" else X @ T) / 2.0
    assert np.abs(Bx).max() < 2.0 ** 50
    pad = 5
    Ah = np.full((order + pad, order), np.nan, order="F")
    r, cidx = np.meshgrid(np.arange(order), np.arange(order), indexing="ij")
    used = (r <= cidx) if uplo == "U" else (r >= cidx)
    if diag == "U":
        used &= r != cidx
    Ah[:order][used] = A[used]
    Al = np.where(np.isnan(Ah), np.nan, 0.0)
    Bh = np.full((m + pad, n), np.nan, order="F")
    Bh[:m] = Bx
    Bl = np.where(np.isnan(Bh), np.nan, 0.0)
    c = datagen.TrsmCase(side, uplo, transa, diag, m, n, (2.0, 0.0),
                         (np.asfortranarray(Ah), np.asfortranarray(Al)),
                         (np.asfortranarray(Bh), np.asfortranarray(Bl)))
    return c, X


@pytest.mark.parametrize("side,uplo,transa,diag", TRSM_VARIANTS)
def test_integer_solution_exact(cuda_lib, side, uplo, transa, diag):
    m, n = (150, 70) if side == "L" else (70, 150)
    c, X = integer_case(side, uplo, transa, diag, m, n, 800)
    xh, xl = gpu_trsm(cuda_lib, c)
    assert np.array_equal(xh, X) and not xl.any()


@pytest.mark.parametrize("side,uplo,transa,diag", TRSM_VARIANTS)
def test_ragged_against_exact_residual_and_oracle(cuda_lib, side, uplo, transa, diag):
    m, n = (150, 70) if side == "L" else (70, 150)
    c = datagen.trsm_case(810, side, uplo, transa, diag, m, n, pad=3)
    got = gpu_trsm(cuda_lib, c)
    assert np.isfinite(got[0]).all()
    assert trsm_residual_over_bound(c, got) <= 1.0
    ref = oracle.dd_trsm(side, uplo, transa, diag, c.alpha, c.A, c.B, m, n)
    ref = (ref[0][:m, :n], ref[1][:m, :n])
    # both solutions have backward error <= 4 (order + 2) 2^-104 on a matrix
    # of condition < 4, so they differ by far less than 2^-90 of the largest
    # solution entry of their column
    diff = np.abs((got[0] - ref[0]) + (got[1] - ref[1]))
    col = np.abs(ref[0]).max(axis=0, keepdims=True)
    assert (diff <= 2.0 ** -90 * col).all()


@pytest.mark.parametrize("side,uplo,transa,diag",
                         [("L", "U", "N", "N"), ("L", "L", "T", "U"), ("R", "U", "T", "N"),
                          ("R", "L", "N", "N")])
def test_larger_sampled(cuda_lib, side, uplo, transa, diag):
    """Orders 700 / 1000 (several recursion levels) on sampled entries."""
    m, n = (1000, 300) if side == "L" else (300, 700)
    c = datagen.trsm_case(820, side, uplo, transa, diag, m, n)
    got = gpu_trsm(cuda_lib, c)
    g = datagen.rng(821)
    rows = g.integers(0, m, 1500)
    cols = g.integers(0, n, 1500)
    # include the last rows/columns (the end of each sweep)
    rows[:50], cols[50:100] = m - 1, n - 1
    assert trsm_residual_over_bound(c, got, rows, cols) <= 1.0


def test_cholesky_factor_of_served_request(cuda_lib):
    """F = G G^T of a served request (condition ~1e20); its dd Cholesky factor
    U (condition ~1e10) solves U^T Y = B then U X = Y within the backward
    bound each time."""
    n = 200
    G, B = datagen.spd_request(830, n)
    Fd = oracle.dd_syrk("U", "N", (1.0, 0.0), G, (0.0, 0.0),
                        (np.zeros((n, n), order="F"), np.zeros((n, n), order="F")))
    fh, fl, info = oracle.dd_potrf("U", Fd)
    assert info == 0
    U = (np.where(np.triu(np.ones((n, n))) > 0, fh, np.nan),
         np.where(np.triu(np.ones((n, n))) > 0, fl, np.nan))
    U = tuple(np.asfortranarray(x) for x in U)
    for transa in "TN":
        c = datagen.TrsmCase("L", "U", transa, "N", n, B[0].shape[1], (1.0, 0.0), U, B)
        got = gpu_trsm(cuda_lib, c)
        assert trsm_residual_over_bound(c, got) <= 1.0
        B = tuple(np.asfortranarray(x) for x in got)


def test_alpha_zero_empty_and_errors(cuda_lib):
    mp = cuda_lib
    c = datagen.trsm_case(840, "L", "U", "N", "N", 40, 30)
    A, B = dev(c.A), dev(c.B)
    nanA = tuple(torch.full_like(x, float("nan")) for x in A)
    mp.mp_dd_Rtrsm("L", "U", "N", "N", 40, 30, (0.0, 0.0), nanA, 40, B, 40)
    xh, xl = host(B)
    assert not xh.any() and not xl.any()
    B = dev(c.B)
    mp.mp_dd_Rtrsm("L", "U", "N", "N", 0, 30, c.alpha, A, 40, B, 40)
    mp.mp_dd_Rtrsm("R", "U", "N", "N", 40, 0, c.alpha, A, 1, B, 40)
    xh, xl = host(B)
    assert np.array_equal(xh, c.B[0]) and np.array_equal(xl, c.B[1])
    bad = [(("X", "U", "N", "N", 40, 30, 40, 40), -1), (("L", "X", "N", "N", 40, 30, 40, 40), -2),
           (("L", "U", "X", "N", 40, 30, 40, 40), -3), (("L", "U", "N", "X", 40, 30, 40, 40), -4),
           (("L", "U", "N", "N", -1, 30, 40, 40), -5), (("L", "U", "N", "N", 40, -1, 40, 40), -6),
           (("L", "U", "N", "N", 40, 30, 39, 40), -9), (("R", "U", "N", "N", 40, 30, 29, 40), -9),
           (("L", "U", "N", "N", 40, 30, 40, 39), -11)]
    for (s, u, t, d, m, n, lda, ldb), code in bad:
        rc = mp.mp_dd_Rtrsm(s, u, t, d, m, n, c.alpha, A, lda, B, ldb, check=False)
        assert rc == code, (s, u, t, d, m, n, lda, ldb, rc)
    # lower-case and 'C' flags are accepted
    B = dev(c.B)
    mp.mp_dd_Rtrsm("l", "u", "c", "n", 40, 30, c.alpha, A, 40, B, 40)


def test_deterministic(cuda_lib):
    c = datagen.trsm_case(850, "R", "L", "T", "N", 90, 260)
    a = gpu_trsm(cuda_lib, c)
    b = gpu_trsm(cuda_lib, c)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("transa", ["N", "T"])
def test_result_independent_of_columns_per_cta(cuda_lib, transa):
    """The solve kernel runs 32, 16, 8 or 4 right-hand-side columns per CTA
    depending on how many columns there are; each column's result is the
    same bits in every configuration."""
    m, wide = 150, 10000
    c = datagen.trsm_case(851, "L", "U", transa, "N", m, wide)
    outs = []
    for n in (6, 2500, 5000, wide):
        B = tuple(np.asfortranarray(P[:, :n]) for P in c.B)
        sub = datagen.TrsmCase(c.side, c.uplo, c.transa, c.diag, m, n, c.alpha, c.A, B)
        outs.append(gpu_trsm(cuda_lib, sub))
    for h, l in outs[1:]:
        assert np.array_equal(h[:, :6], outs[0][0]) and np.array_equal(l[:, :6], outs[0][1])


@pytest.mark.parametrize("side,uplo,transa,diag",
                         [("L", "U", "N", "N"), ("L", "L", "N", "U"), ("R", "U", "T", "N"),
                          ("R", "L", "T", "U")])
@pytest.mark.parametrize("form", ["plain", "scaled", "nonfinite"])
def test_tensor_core_updates(cuda_lib, side, uplo, transa, diag, form):
    """Orders whose updates run in residue form (700 with 900 right-hand
    sides): the backward error stays within a tenth of the bound of
    substitution (per entry at most five updates of 6u^2 and 64 steps of 8u^2
    against 16 * 702 u^2: 0.05).  "scaled": rows of the triangle and of B over
    120 binades, so that updates need wider operands or the FP64 pipe.
    "nonfinite": an infinity in one column (row) of B spoils that one only."""
    m, n = (700, 900) if side == "L" else (900, 700)
    c = datagen.trsm_case(860, side, uplo, transa, diag, m, n)
    g = datagen.rng(861)
    order = 700
    if form == "scaled":
        # D A D^-1 keeps the triangle's diagonal; B scaled along the other side
        e = g.integers(-30, 31, order)
        f = np.ldexp(1.0, e)
        for P in c.A:
            P[:order] *= f[:, None] / f[None, :]
        h = np.ldexp(1.0, g.integers(-60, 61, 900))
        for P in c.B:
            P[:m] *= h[None, :] if side == "L" else h[:, None]
    if form == "nonfinite":
        c.B[0][(5, 7) if side == "L" else (7, 5)] = np.inf
    X = gpu_trsm(cuda_lib, c)
    keep = np.arange(900) != 7
    if form == "nonfinite":
        bad = X[0][:, 7] if side == "L" else X[0][7]
        assert not np.isfinite(bad).all()
        rest = X[0][:, keep] if side == "L" else X[0][keep]
        assert np.isfinite(rest).all()
    rows, cols = g.integers(0, m, 1200), g.integers(0, n, 1200)
    rows[:40], cols[40:80] = m - 1, n - 1
    rows[80:120], cols[120:160] = 0, 0
    if form == "nonfinite":
        ok = (cols if side == "L" else rows) != 7
        rows, cols = rows[ok], cols[ok]
        for P in (*c.B, *X):
            P[~np.isfinite(P)] = 0.0
    assert trsm_residual_over_bound(c, X, rows, cols) <= 0.1


def test_updates_are_not_in_the_phase_log(cuda_lib):
    """The phase log holds the split-precision calls, not the tensor-core
    updates that Rtrsm, Rgetrf and Rgetrs make between them (order 512 with
    512 right-hand sides: the 256 x 512 x 256 update of a solve, 471 us on the
    FP64 pipe by the launch's count, runs in residue form)."""
    mp = cuda_lib
    n = 512
    c = datagen.trsm_case(862, "L", "L", "N", "N", n, n)
    A, B = dev(c.A), dev(c.B)
    g = datagen.rng(863)
    F, P, Q = (dev(datagen.dd_matrix(g, n, n)) for _ in range(3))
    ipiv = torch.empty(n, dtype=torch.int64, device="cuda")
    info = torch.empty(1, dtype=torch.int64, device="cuda")
    ws = mp.workspace(mp.mp_dd_Rgemm_crt_workspace(64, 64, 64))

    def product():
        mp.mp_dd_Rgemm_crt("N", "N", 64, 64, 64, (1.0, 0.0), P, n, P, n, (0.0, 0.0), Q, n, ws,
                           ws.numel())

    mp.mp_dd_sliced_timing(True)
    try:
        product()
        mp.mp_dd_Rtrsm("L", "L", "N", "N", n, n, c.alpha, A, n, B, n)
        product()
        mp.mp_dd_Rgetrf(n, n, F, n, ipiv, info)
        mp.mp_dd_Rgetrs("N", n, n, F, n, ipiv, B, n)
        log = mp.mp_dd_sliced_phase_log()
    finally:
        mp.mp_dd_sliced_timing(False)
    assert len(log) == 2 and all(t > 0 for row in log for t in row)


@pytest.mark.parametrize("side,uplo,transa", [("L", "U", "T"), ("R", "L", "N")])
def test_right_hand_sides_alone_and_with_others(cuda_lib, side, uplo, transa):
    """A right-hand side solved with 95, 96 or 640 others at order 320: the
    updates take the FP64 pipe or the residue form by the number of columns, so
    the low bits may differ, and each solution meets the bound of substitution
    (320 steps of at most 8u^2 and a division of 20u^2 against 16 * 322 u^2:
    0.51).  Up to 95 columns every update is on the FP64 pipe and the bits are
    the same."""
    order, wide = 320, 640
    m, n = (order, wide) if side == "L" else (wide, order)
    c = datagen.trsm_case(864, side, uplo, transa, "N", m, n)
    g = datagen.rng(865)
    outs = {}
    for w in (6, 95, 96, wide):
        B = tuple(np.asfortranarray(P[:, :w] if side == "L" else P[:w]) for P in c.B)
        sub = datagen.TrsmCase(side, uplo, transa, "N", *((m, w) if side == "L" else (w, n)),
                               c.alpha, c.A, B)
        X = gpu_trsm(cuda_lib, sub)
        rows, cols = g.integers(0, sub.m, 400), g.integers(0, sub.n, 400)
        if side == "L":
            cols[:200] %= 6
        else:
            rows[:200] %= 6
        assert trsm_residual_over_bound(sub, X, rows, cols) <= 0.51, w
        outs[w] = tuple(x[:, :6] if side == "L" else x[:6] for x in X)
    for a, b in zip(outs[6], outs[95]):
        assert np.array_equal(a, b)


def test_updates_in_blocks_of_the_scratch_limit(cuda_lib):
    """X op(A) = alpha B of order 512 with 160000 rows of B: the 160000 x 256 x
    256 update's workspace is above 4 GiB, so it runs in two blocks of at most
    80128 rows.  The rows at both ends and on either side of the border meet a
    tenth of the bound of substitution (three updates of 6u^2 and 64 steps of
    8u^2 against 16 * 514 u^2: 0.065)."""
    mp = cuda_lib
    m, n = 160000, 512
    assert mp.mp_dd_Rgemm_crt_workspace(m, 256, 256) > 4 << 30
    assert mp.mp_dd_Rgemm_crt_workspace(80128, 256, 256) <= 4 << 30
    c = datagen.trsm_case(866, "R", "U", "N", "N", 8, n)
    gen = torch.Generator(device="cuda").manual_seed(867)
    hi, lo = (torch.empty(n, m, dtype=torch.float64, device="cuda").uniform_(-1, 1, generator=gen)
              for _ in range(2))
    lo *= hi * 2.0 ** -54
    rows = np.r_[0:40, 80108:80148, m - 40:m]
    at = torch.from_numpy(rows).cuda()

    def picked():
        return tuple(np.asfortranarray(x[:, at].cpu().numpy().T) for x in (hi, lo))

    c.B, c.m = picked(), len(rows)
    mp.mp_dd_Rtrsm("R", "U", "N", "N", m, n, c.alpha, dev(c.A), n, (hi, lo), m)
    torch.cuda.synchronize()
    g = datagen.rng(868)
    r = np.tile(np.arange(len(rows)), 10)
    cols = np.where(g.random(len(r)) < 0.7, g.integers(256, n, len(r)), g.integers(0, n, len(r)))
    assert trsm_residual_over_bound(c, picked(), r, cols) <= 0.1


def test_residue_updates_round_no_worse_than_the_fp64_pipe(cuda_lib):
    """150 right-hand sides together (updates in residue form) and 75 at a time
    (every update on the FP64 pipe), order 1300 with a unit diagonal and small
    entries, where alpha B plus an update makes most of the error: the
    residual's mean square relative to |A||X| + |alpha B|, formed in quad-double,
    is no larger (0.5 % for the difference of two samples of 195000 entries with
    the same final roundings; a sum with more roundings gave 1.019 times it)."""
    mp = cuda_lib
    m, w = 1300, 150
    gen = torch.Generator(device="cuda").manual_seed(869)

    def rand(r, c):
        return torch.empty(c, r, dtype=torch.float64, device="cuda").uniform_(-1, 1, generator=gen).t()

    def dd(hi):
        return hi, hi * rand(*hi.shape) * 2.0 ** -54

    def planes(x):
        zero = torch.zeros_like(x[0].t().contiguous()).t()
        return [*(p.t().clone().t() for p in x), zero, zero.clone()]

    A = dd((torch.triu(rand(m, m), 1) / m).t().contiguous().t())
    B = dd(rand(m, w))
    alpha = datagen.dd_scalar(datagen.rng(870))
    T = (A[0] + torch.eye(m, dtype=torch.float64, device="cuda"), A[1])
    rms = []
    for step in (w, 75):
        X = tuple(p.t().clone().t() for p in B)
        for j in range(0, w, step):
            part = tuple(p[:, j:j + step] for p in X)
            mp.mp_dd_Rtrsm("L", "U", "N", "U", m, step, alpha, A, m, part, m)
        R = planes(B)
        mp.mp_qd_Rgemm("N", "N", m, w, m, (1.0,), planes(T), m, planes(X), m,
                       (-alpha[0], -alpha[1]), R, m)
        scale = T[0].abs() @ X[0].abs() + alpha[0] * B[0].abs()
        rms.append((R[0] / scale).pow(2).mean().sqrt().item())
    assert rms[0] <= 1.005 * rms[1]
