"""The work that users of this library call it for, as measurable cases.

Every case goes through the public entry points of ``paper_2109_13406_gb300``
on column-major dd (or qd) planes that are on the GPU.  ``listed`` holds one
case of each kind of use, from the smallest calls to the largest; ``draw``
spreads the same kinds over their whole ranges of sizes.

Inputs follow the recipes of the tests and the benchmark: dd entries hi ~
U(-1, 1) with lo = hi 2^-53 U(-1, 1), renormalised; dd scalars in [0.5, 2];
grouped problem sizes log-uniform in 16 .. 512; symmetric positive definite
matrices M M^T / k + I; LU matrices with U(-1, 1) entries.  Calls that update
a matrix in place first copy the caller's matrix into the buffer they write.
"""
import math

import torch

import paper_2109_13406_gb300 as mp
from paper_2109_13406_gb300 import grouped


def listed():
    return [
        # The smallest call: one tile row of a hand-sized product (launch and latency).
        dict(name="gemm_nn_96x80x70", kind="gemm", ta="N", tb="N", m=96, n=80, k=70, pad=3, beta=False),
        # An ordinary FP64-pipe product: odd sizes, leading dimensions with padding,
        # a transposed operand, C updated.
        dict(name="gemm_tn_1101x700x905", kind="gemm", ta="T", tb="N", m=1101, n=700, k=905, pad=5, beta=True),
        # One triangle of a Gram matrix on the FP64 pipe.
        dict(name="syrk_un_1024", kind="syrk", uplo="U", trans="N", n=1024, k=1024, pad=0, beta=False),
        # Quad-double, where dd is not enough.
        dict(name="qd_nt_331x300x257", kind="qd", ta="N", tb="T", m=331, n=300, k=257),
        # A small certified split-precision product: many short launches.
        dict(name="crt_nn_512", kind="crt", ta="N", tb="N", m=512, n=512, k=512, pad=0, beta=False),
        # An ordinary one: odd sizes, a transposed operand, C updated.
        dict(name="crt_tn_1501x2777x1999", kind="crt", ta="T", tb="N", m=1501, n=2777, k=1999, pad=1, beta=True),
        # The headline product of the benchmark.
        dict(name="crt_nn_8192", kind="crt", ta="N", tb="N", m=8192, n=8192, k=8192, pad=0, beta=True),
        # Its Rsyrk, at an ordinary size.
        dict(name="syrk_crt_un_4096", kind="syrk_crt", uplo="U", trans="N", n=4096, k=4096, pad=0, beta=True),
        # The digit form on badly scaled rows and columns.
        dict(name="sliced_nn_2048", kind="sliced", ta="N", tb="N", m=2048, n=2048, k=2048, pad=0, beta=False),
        # Many small uneven products in one launch, as a batched program keeps them planned.
        dict(name="grouped_512", kind="grouped", count=512),
        # A positive definite system: factor on the tensor cores, then solve.
        dict(name="cholesky_solve_3000", kind="cholesky", n=3000, nrhs=4),
        # A general system with many right-hand sides: LU, then triangular solves.
        dict(name="lu_solve_1536", kind="lu", n=1536, nrhs=500),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["gemm", "syrk", "qd", "crt", "crt", "syrk_crt", "sliced", "grouped", "cholesky", "lu", "trsm"])
    flag = lambda: rng.choice(["N", "T"])  # noqa: E731
    if kind in ("gemm", "crt", "sliced"):
        lo, hi = {"gemm": (32, 1400), "crt": (96, 8000), "sliced": (96, 3000)}[kind]
        return dict(kind=kind, ta=flag(), tb=flag(), m=_log(rng, lo, hi), n=_log(rng, lo, hi), k=_log(rng, lo, hi),
                    pad=rng.choice([0, 0, 1, 4, 7]), beta=rng.random() < 0.5)
    if kind in ("syrk", "syrk_crt"):
        lo, hi = {"syrk": (48, 1400), "syrk_crt": (128, 8000)}[kind]
        return dict(kind=kind, uplo=rng.choice(["U", "L"]), trans=flag(), n=_log(rng, lo, hi), k=_log(rng, lo, hi),
                    pad=rng.choice([0, 0, 1, 6]), beta=rng.random() < 0.5)
    if kind == "qd":
        return dict(kind=kind, ta=flag(), tb=flag(), m=_log(rng, 32, 500), n=_log(rng, 32, 500), k=_log(rng, 32, 500))
    if kind == "grouped":
        return dict(kind=kind, count=_log(rng, 32, 700))
    if kind == "cholesky":
        return dict(kind=kind, n=_log(rng, 200, 4500), nrhs=rng.choice([1, 4, 16, 65]))
    if kind == "lu":
        return dict(kind=kind, n=_log(rng, 128, 2300), nrhs=_log(rng, 1, 900))
    return dict(kind="trsm", side=rng.choice(["L", "R"]), uplo=rng.choice(["U", "L"]), ta=flag(),
                diag=rng.choice(["N", "U"]), m=_log(rng, 64, 2300), n=_log(rng, 64, 2300))


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _rand(g, rows, cols, ld):
    """Column-major rows x cols view with leading dimension ld, U(-1, 1)."""
    return torch.empty((cols, ld), dtype=torch.float64, device="cuda").uniform_(-1, 1, generator=g).t()[:rows]


def _two(hi, lo):
    s = hi + lo
    return s, lo - (s - hi)


def _dd(g, rows, cols, pad=0):
    hi = _rand(g, rows, cols, rows + pad)
    return _two(hi, hi * _rand(g, rows, cols, rows + pad) * 2.0 ** -53)


def _like_dd(g, hi):
    """hi (column major) with a lo plane drawn as in _dd."""
    return _two(hi, hi * _rand(g, hi.shape[0], hi.shape[1], hi.shape[0]) * 2.0 ** -53)


def _scalar(g, low=0.5, high=2.0):
    u = torch.empty(2, dtype=torch.float64, device="cuda").uniform_(0, 1, generator=g).tolist()
    hi = low + (high - low) * u[0]
    lo = hi * 2.0 ** -53 * (2.0 * u[1] - 1.0)
    return hi + lo, lo - ((hi + lo) - hi)


def _scale(pair, exponents, dim):
    f = torch.pow(2.0, exponents.to(torch.float64))
    f = f[:, None] if dim == 0 else f[None, :]
    return tuple(x * f for x in pair)


def _empty(rows, cols, pad=0):
    return mp.dd_empty(rows, cols, rows + pad)


def _copy(dst, src):
    for d, s in zip(dst, src):
        d.copy_(s)


def _ld(pair):
    return pair[0].stride(1) if pair[0].shape[1] > 1 else max(1, pair[0].shape[0])


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    c = dict(case)
    kind, s = c["kind"], {"case": c}
    if kind in ("gemm", "crt", "sliced"):
        m, n, k, pad = c["m"], c["n"], c["k"], c["pad"]
        s["A"] = _dd(g, *((k, m) if c["ta"] == "T" else (m, k)), pad)
        s["B"] = _dd(g, *((n, k) if c["tb"] == "T" else (k, n)), pad)
        if kind == "sliced":   # rows of op(A) and columns of op(B) over 60 binades
            ea = torch.randint(-30, 31, (m,), device="cuda", generator=g)
            eb = torch.randint(-30, 31, (n,), device="cuda", generator=g)
            s["A"] = _scale(s["A"], ea, 1 if c["ta"] == "T" else 0)
            s["B"] = _scale(s["B"], eb, 0 if c["tb"] == "T" else 1)
        s["alpha"], s["beta"] = _scalar(g), (_scalar(g) if c["beta"] else (0.0, 0.0))
        s["C"] = _empty(m, n, pad)
        if c["beta"]:
            s["C0"] = _dd(g, m, n, pad)
        if kind == "crt":
            s["ws"] = mp.workspace(mp.mp_dd_Rgemm_crt_workspace(m, n, k))
        if kind == "sliced":
            s["ws"] = mp.workspace(mp.mp_dd_Rgemm_sliced_workspace(m, n, k, 0))
    elif kind in ("syrk", "syrk_crt"):
        n, k, pad = c["n"], c["k"], c["pad"]
        s["A"] = _dd(g, *((k, n) if c["trans"] == "T" else (n, k)), pad)
        s["alpha"], s["beta"] = _scalar(g), (_scalar(g) if c["beta"] else (0.0, 0.0))
        s["C"] = _empty(n, n, pad)
        s["C0"] = _dd(g, n, n, pad)
        _copy(s["C"], s["C0"])
        if kind == "syrk_crt":
            s["ws"] = mp.workspace(mp.mp_dd_Rsyrk_crt_workspace(n, k))
    elif kind == "qd":
        m, n, k = c["m"], c["n"], c["k"]

        def qd(rows, cols):
            x = [_rand(g, rows, cols, rows)]
            for _ in range(3):
                x.append(x[-1] * _rand(g, rows, cols, rows) * 2.0 ** -53)
            for _ in range(2):
                for t in range(3):
                    x[t], x[t + 1] = _two(x[t], x[t + 1])
            return x

        s["A"] = qd(*((k, m) if c["ta"] == "T" else (m, k)))
        s["B"] = qd(*((n, k) if c["tb"] == "T" else (k, n)))
        s["C"] = _empty(m, n) + _empty(m, n)
    elif kind == "grouped":
        r = torch.empty((c["count"], 3), dtype=torch.float64).uniform_(
            math.log(16), math.log(512), generator=torch.Generator().manual_seed(c["count"]))
        sizes = [tuple(int(round(math.exp(v))) for v in row) for row in r.tolist()]
        total = sum(m * n for m, n, _ in sizes)
        s["out"] = tuple(torch.empty(total, dtype=torch.float64, device="cuda") for _ in range(2))
        problems, at = [], 0
        for m, n, k in sizes:
            C = tuple(o[at:at + m * n].view(n, m).t() for o in s["out"])
            at += m * n
            problems.append(("N", "N", m, n, k, (1.0, 0.0), _dd(g, m, k), _dd(g, k, n), (0.0, 0.0), C))
        s["problems"], s["plan"] = problems, grouped.GroupedGemm(problems)
    elif kind == "cholesky":
        n = c["n"]
        M = _rand(g, n, n, n)
        A = M @ M.t() / n
        A.diagonal().add_(1.0)
        A = torch.triu(A) + torch.triu(A, 1).t()
        s["A0"] = _like_dd(g, A.t().contiguous().t())
        s["B0"] = _dd(g, n, c["nrhs"])
        s["A"], s["B"] = _empty(n, n), _empty(n, c["nrhs"])
        s["info"] = torch.zeros(1, dtype=torch.int64, device="cuda")
        s["ws"] = mp.workspace(mp.mp_dd_Rpotrf_crt_workspace(n))
    elif kind == "lu":
        n = c["n"]
        s["A0"], s["B0"] = _dd(g, n, n), _dd(g, n, c["nrhs"])
        s["A"], s["B"] = _empty(n, n), _empty(n, c["nrhs"])
        s["ipiv"] = torch.zeros(n, dtype=torch.int64, device="cuda")
        s["info"] = torch.zeros(1, dtype=torch.int64, device="cuda")
    elif kind == "trsm":
        m, n = c["m"], c["n"]
        q = m if c["side"] == "L" else n
        hi = _rand(g, q, q, q)
        hi = hi / q if c["diag"] == "U" else hi + torch.diag(torch.sign(hi.diagonal()) * (q - 1))
        s["A"] = _like_dd(g, hi.t().contiguous().t())
        s["alpha"], s["B0"], s["B"] = _scalar(g), _dd(g, m, n), _empty(m, n)
    else:
        raise ValueError(kind)
    return s


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind in ("gemm", "crt", "sliced"):
        if c["beta"]:
            _copy(s["C"], s["C0"])
        A, B, C = s["A"], s["B"], s["C"]
        args = (c["ta"], c["tb"], c["m"], c["n"], c["k"], s["alpha"], A, _ld(A), B, _ld(B), s["beta"], C, _ld(C))
        if kind == "gemm":
            mp.mp_dd_Rgemm(*args)
        elif kind == "crt":
            mp.mp_dd_Rgemm_crt(*args, s["ws"], s["ws"].numel())
        else:
            mp.mp_dd_Rgemm_sliced(*args, 0, s["ws"], s["ws"].numel())
        return C
    if kind in ("syrk", "syrk_crt"):
        if c["beta"]:
            _copy(s["C"], s["C0"])
        A, C = s["A"], s["C"]
        args = (c["uplo"], c["trans"], c["n"], c["k"], s["alpha"], A, _ld(A), s["beta"], C, _ld(C))
        if kind == "syrk":
            mp.mp_dd_Rsyrk(*args)
        else:
            mp.mp_dd_Rsyrk_crt(*args, s["ws"], s["ws"].numel())
        return C
    if kind == "qd":
        A, B, C = s["A"], s["B"], s["C"]
        mp.mp_qd_Rgemm(c["ta"], c["tb"], c["m"], c["n"], c["k"], (1.0,), A, _ld(A), B, _ld(B), (0.0,), C, _ld(C))
        return C
    if kind == "grouped":
        s["plan"].run()
        return s["out"]
    if kind == "cholesky":
        n, A, B = c["n"], s["A"], s["B"]
        _copy(A, s["A0"])
        _copy(B, s["B0"])
        mp.mp_dd_Rpotrf_crt("U", n, A, n, s["info"], s["ws"], s["ws"].numel())
        mp.mp_dd_Rpotrs("U", n, c["nrhs"], A, n, B, n, s["info"])
        return A, B, s["info"]
    if kind == "lu":
        n, A, B = c["n"], s["A"], s["B"]
        _copy(A, s["A0"])
        _copy(B, s["B0"])
        mp.mp_dd_Rgetrf(n, n, A, n, s["ipiv"], s["info"])
        mp.mp_dd_Rgetrs("N", n, c["nrhs"], A, n, s["ipiv"], B, n)
        return A, B, s["ipiv"], s["info"]
    A, B = s["A"], s["B"]
    _copy(B, s["B0"])
    mp.mp_dd_Rtrsm(c["side"], c["uplo"], c["ta"], c["diag"], c["m"], c["n"], s["alpha"], A, _ld(A), B, _ld(B))
    return B


def _sizes(case):
    """(m, n, k) of each product of a product case."""
    if case["kind"] in ("syrk", "syrk_crt"):
        return case["n"], case["n"], case["k"]
    return case["m"], case["n"], case["k"]


def work(case):
    """dd (qd) operands at 16 (32) bytes an entry, and the routines' usual
    operation counts with one dd (qd) operation as one flop."""
    kind = case["kind"]
    if kind in ("gemm", "crt", "sliced", "qd"):
        m, n, k = _sizes(case)
        reads_c = 1 if case.get("beta") else 0
        return {"bytes": (32 if kind == "qd" else 16) * (m * k + k * n + (1 + reads_c) * m * n), "flops": 2 * m * n * k}
    if kind in ("syrk", "syrk_crt"):
        n, k = case["n"], case["k"]
        tri = n * (n + 1) // 2
        return {"bytes": 16 * (n * k + (2 if case["beta"] else 1) * tri), "flops": 2 * k * tri}
    if kind == "grouped":
        r = torch.empty((case["count"], 3), dtype=torch.float64).uniform_(
            math.log(16), math.log(512), generator=torch.Generator().manual_seed(case["count"]))
        sizes = [tuple(int(round(math.exp(v))) for v in row) for row in r.tolist()]
        return {"bytes": sum(16 * (m * k + k * n + m * n) for m, n, k in sizes),
                "flops": sum(2 * m * n * k for m, n, k in sizes)}
    if kind == "cholesky":
        n, r = case["n"], case["nrhs"]
        return {"bytes": 16 * (n * (n + 1) + 2 * n * r), "flops": n ** 3 // 3 + 2 * n * n * r}
    if kind == "lu":
        n, r = case["n"], case["nrhs"]
        return {"bytes": 16 * (2 * n * n + 2 * n * r), "flops": 2 * n ** 3 // 3 + 2 * n * n * r}
    m, n = case["m"], case["n"]
    q, r = (m, n) if case["side"] == "L" else (n, m)
    return {"bytes": 16 * (q * (q + 1) // 2 + 2 * m * n), "flops": q * q * r}


# --------------------------------------------------------------------------
# the same results in 64 bits
# --------------------------------------------------------------------------

def _sum(hi, lo, p):
    """(hi, lo) + p, p a float64 tensor."""
    s = hi + p
    b = s - hi
    return _two(s, lo + ((hi - (s - b)) + (p - b)))


def _times(x, scalar):
    """dd tensor times a dd scalar (products split by Veltkamp and Dekker)."""
    def split(v):
        t = 134217729.0 * v
        h = t - (t - v)
        return h, v - h

    (a, b), (sh, sl) = x, scalar
    p = a * sh
    ah, al = split(a)
    th, tl = split(torch.tensor(sh, dtype=torch.float64, device=a.device))
    e = ((ah * th - p) + ah * tl + al * th) + al * tl
    return _two(p, e + (a * sl + b * sh))


def _slices(x, dim, bits, count):
    """x = sum of count slices whose entries are multiples of one unit per
    row (dim 1) or column (dim 0) and at most 2^bits units."""
    hi, lo = x
    top = torch.amax(torch.abs(hi), dim=dim, keepdim=True)
    unit = torch.where(top > 0, torch.pow(2.0, torch.floor(torch.log2(torch.clamp(top, min=1e-300))) + 2 - bits), torch.ones_like(top))
    out = []
    for _ in range(count):
        q = torch.round(hi / unit) * unit
        out.append(q)
        hi, lo = _two(hi - q, lo)
        unit = unit * 2.0 ** -bits
    return out


def _product(a, b, block=1024):
    """The dd product of dd tensors from float64 matmuls without rounding
    error, block by block (a library may compute a large float64 matmul by
    other means, which are not exact for integers)."""
    m, k, n = a[0].shape[0], a[0].shape[1], b[0].shape[1]
    bits = int((52 - math.ceil(math.log2(max(2, min(block, k))))) // 2)
    count = -(-118 // bits)
    sa, sb = _slices(a, 1, bits, count), _slices(b, 0, bits, count)
    hi = torch.zeros((m, n), dtype=torch.float64, device=a[0].device)
    lo = torch.zeros_like(hi)
    for i in range(0, m, block):
        for j in range(0, n, block):
            r = hi[i:i + block, j:j + block], lo[i:i + block, j:j + block]
            for l in range(0, k, block):
                for t in range(count):
                    for u in range(t + 1):
                        r = _sum(*r, sa[u][i:i + block, l:l + block] @ sb[t - u][l:l + block, j:j + block])
            hi[i:i + block, j:j + block], lo[i:i + block, j:j + block] = r
    return hi, lo


def exact(case, seed):
    s = prepare(case, seed)
    c, kind = s["case"], s["case"]["kind"]
    op = lambda x, t: tuple(v.t() for v in x) if t == "T" else x  # noqa: E731
    if kind in ("gemm", "crt", "sliced", "syrk", "syrk_crt"):
        if kind in ("syrk", "syrk_crt"):
            a = op(s["A"], c["trans"])
            b = tuple(v.t() for v in a)
        else:
            a, b = op(s["A"], c["ta"]), op(s["B"], c["tb"])
        m, n, k = _sizes(c)
        whole = m * n * k <= 2 ** 33
        if whole:
            r = _times(_product(a, b), s["alpha"])
            if c["beta"]:
                t = _times(s["C0"], s["beta"])
                r = _sum(*_sum(*r, t[1]), t[0])
        else:
            hi = s["alpha"][0] * (a[0] @ b[0])
            r = (hi + s["beta"][0] * s["C0"][0] if c["beta"] else hi, None)
        if kind in ("syrk", "syrk_crt"):
            keep = torch.ones((n, n), dtype=torch.bool, device="cuda")
            keep = torch.triu(keep) if c["uplo"] == "U" else torch.tril(keep)
            r = tuple(None if x is None else torch.where(keep, x, y) for x, y in zip(r, s["C0"]))
        return r
    if kind == "qd":
        return [op(s["A"], c["ta"])[0] @ op(s["B"], c["tb"])[0], None, None, None]
    if kind == "grouped":
        parts = [_product(A, B) for (_, _, _, _, _, _, A, B, _, _) in s["problems"]]
        return tuple(torch.cat([p[q].t().reshape(-1) for p in parts]) for q in range(2))
    if kind == "cholesky":
        # the factor in the upper triangle, the matrix below it
        U = torch.linalg.cholesky(s["A0"][0], upper=True)
        X = torch.cholesky_solve(s["B0"][0], U, upper=True)
        return (torch.triu(U) + torch.tril(s["A0"][0], -1), None), (X, None), None
    if kind == "lu":
        F, _ = torch.linalg.lu_factor(s["A0"][0])
        return (F, None), (torch.linalg.solve(s["A0"][0], s["B0"][0]), None), None, None
    A = torch.triu(s["A"][0]) if c["uplo"] == "U" else torch.tril(s["A"][0])
    upper = (c["uplo"] == "U") != (c["ta"] == "T")
    X = torch.linalg.solve_triangular(A.t() if c["ta"] == "T" else A, s["alpha"][0] * s["B0"][0], upper=upper,
                                      left=c["side"] == "L", unitriangular=c["diag"] == "U")
    return X, None
