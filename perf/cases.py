"""What a program does with this library, as cases that can be timed.

Each case is one call, or one factorization with the solve that follows it,
through the binding's public entry points.  listed() holds the standing cases,
draw() gives further ones of the same ranges.  The sizes are those of the
repository's own configurations, tests and benchmark (n = 32768 for the large
LU, 16384 x 16384 x 256 for its trailing update, n in [64, 1024] for the
batched systems) or generic odd ones.
"""
import math
import os

import torch

import paper_2509_23565_gb300
from paper_2509_23565_gb300.binding import ColMajor, Emul

_EMUL = None      # the one handle a program keeps


def _handle():
    global _EMUL
    if _EMUL is None:
        _EMUL = Emul()
        _EMUL.selector_load(os.path.join(os.path.dirname(paper_2509_23565_gb300.__file__), "selector_weights.bin"))
    return _EMUL


def listed():
    return [
        # the smallest products, as the inner steps of a small blocked algorithm
        # make them one after another: latency and launches count
        {"name": "gemm_small", "kind": "gemm", "m": 64, "n": 64, "k": 64, "s": 7, "alpha": 1.0, "beta": 0.0,
         "pad": 0, "r": 0.0},
        # an ordinary BLAS call with ragged sizes, leading dimensions larger
        # than the rows, general alpha and beta, entries of several magnitudes
        {"name": "gemm_ragged", "kind": "gemm", "m": 777, "n": 1001, "k": 333, "s": 6, "alpha": 1.5, "beta": 0.5,
         "pad": 3, "r": 4.0},
        # a square matrix product (the DGEMM sweep's 4096)
        {"name": "gemm_square", "kind": "gemm", "m": 4096, "n": 4096, "k": 4096, "s": 7, "alpha": 1.0, "beta": 0.0,
         "pad": 0, "r": 0.0},
        # the trailing update of a large factorization
        {"name": "gemm_update", "kind": "gemm", "m": 16384, "n": 16384, "k": 256, "s": 7, "alpha": -1.0, "beta": 1.0,
         "pad": 0, "r": 0.0},
        # the same update with the safe slice count that wide-range data needs
        {"name": "gemm_update_s8", "kind": "gemm", "m": 8192, "n": 8192, "k": 256, "s": 8, "alpha": -1.0, "beta": 1.0,
         "pad": 0, "r": 4.0},
        # a small dense system, one right-hand side: the panel's latency
        {"name": "lu_small", "kind": "lu", "n": 500, "nb": 0, "s": 7, "nrhs": 1, "r": 0.0},
        # an ordinary system of odd size with a few right-hand sides
        {"name": "lu_mid", "kind": "lu", "n": 4001, "nb": 128, "s": 7, "nrhs": 8, "r": 0.0},
        # the large LU and solve that the library is built for
        {"name": "lu_large", "kind": "lu", "n": 32768, "nb": 256, "s": 7, "nrhs": 1, "r": 0.0},
        # the slice count left to the selector, on wide-range data
        {"name": "lu_selected", "kind": "lu", "n": 6000, "nb": 256, "s": 0, "nrhs": 1, "r": 2.0},
        # a covariance-like SPD system
        {"name": "chol", "kind": "chol", "n": 12000, "nb": 256, "s": 7, "nrhs": 1},
        # a diagonally dominant system factored without pivoting, default block
        {"name": "lu_nopiv", "kind": "nopiv", "n": 6144, "nb": 0, "s": 7, "nrhs": 1},
        # many uneven systems at once, n log-uniform, half of them wide-range
        {"name": "batched", "kind": "batched", "count": 1024, "lo": 64, "hi": 1024, "r": 8.0},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["gemm", "gemm", "gemm", "gemm", "lu", "lu", "chol", "nopiv", "batched"])
    if kind == "gemm":
        while True:
            m, n, k = _log(rng, 33, 16384), _log(rng, 33, 16384), _log(rng, 33, 4096)
            if m * n * k <= 4096 ** 3:
                break
        alpha, beta = rng.choice([(1.0, 0.0), (-1.0, 1.0), (1.5, 0.5)])
        return {"kind": kind, "m": m, "n": n, "k": k, "s": rng.choice([3, 5, 6, 7, 7, 8]), "alpha": alpha,
                "beta": beta, "pad": rng.choice([0, 0, 1, 8]), "r": rng.choice([0.0, 4.0])}
    if kind == "lu":
        s = rng.choice([0, 6, 7, 7, 8])
        return {"kind": kind, "n": _log(rng, 200, 12000), "nb": rng.choice([0, 64, 256, 512]), "s": s,
                "nrhs": rng.choice([1, 1, 3, 16]), "r": rng.choice([0.0, 2.0])}
    if kind == "chol":
        return {"kind": kind, "n": _log(rng, 300, 16384), "nb": rng.choice([0, 64, 256, 512]),
                "s": rng.choice([6, 7, 8]), "nrhs": rng.choice([1, 1, 4])}
    if kind == "nopiv":
        return {"kind": kind, "n": _log(rng, 300, 8192), "nb": rng.choice([0, 64, 256, 512]),
                "s": rng.choice([6, 7, 8]), "nrhs": rng.choice([1, 1, 4])}
    lo = rng.choice([64, 100, 200])
    return {"kind": kind, "count": _log(rng, 16, 1024), "lo": lo, "hi": _log(rng, 2 * lo, 1024),
            "r": rng.choice([0.0, 8.0])}


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _entries(g, cols, rows, r):
    """u, or u 10^e with e ~ U(-r, r), u ~ U(-1, 1): a column-major store (row j is column j)."""
    x = torch.rand((cols, rows), generator=g, device="cuda", dtype=torch.float64).mul_(2.0).sub_(1.0)
    if r:
        x *= torch.pow(10.0, torch.rand((cols, rows), generator=g, device="cuda", dtype=torch.float64) * (2 * r) - r)
    return x


def _matrix(case, seed):
    """The n x n matrix of a factorization, column-major."""
    g, n = _gen(seed), case["n"]
    if case["kind"] == "chol":      # factor model: a low-rank part and a diagonal
        u = torch.randn((n, 64), generator=g, device="cuda", dtype=torch.float64) / 8.0
        d = torch.rand(n, generator=g, device="cuda", dtype=torch.float64) + 0.5
        a = u @ u.T
        a.diagonal().add_(d)
        return a, g
    a = _entries(g, n, n, case.get("r", 0.0))
    if case["kind"] == "nopiv":
        a.diagonal().fill_(float(n))
    return a, g


def _batch(case, seed):
    """Systems one after another in one buffer: sizes (the case's, log-uniform
    and in no order), matrices, right-hand sides."""
    g = _gen(seed)
    lo, hi = math.log(case["lo"]), math.log(case["hi"] + 1)
    u = [(i * 0.6180339887498949) % 1.0 for i in range(1, case["count"] + 1)]
    ns = [min(case["hi"], max(case["lo"], int(math.exp(lo + (hi - lo) * v)))) for v in u]
    a = _entries(g, 1, sum(n * n for n in ns), 0.0)[0]
    mats, o = [], 0
    for i, n in enumerate(ns):
        m = a[o:o + n * n].view(n, n)
        if case["r"] and i % 2:
            m *= torch.pow(10.0, torch.rand((n, n), generator=g, device="cuda", dtype=torch.float64)
                           * (2 * case["r"]) - case["r"])
        mats.append(m)
        o += n * n
    return ns, mats, _entries(g, 1, sum(ns), 0.0)[0]


def prepare(case, seed):
    st = {"case": case, "emul": _handle()}
    if case["kind"] == "gemm":
        g, p = _gen(seed), case["pad"]
        m, n, k = case["m"], case["n"], case["k"]
        st["A"] = ColMajor(_entries(g, k, m + p, case["r"]), m, k)
        st["B"] = ColMajor(_entries(g, n, k + p, case["r"]), k, n)
        st["C"] = ColMajor(_entries(g, n, m + p, 0.0), m, n)
    elif case["kind"] == "batched":
        ns, mats, b = _batch(case, seed)
        st["b0"], st["x"] = b, torch.empty_like(b)
        st["As"] = [ColMajor(m, n, n) for m, n in zip(mats, ns)]
        st["bs"], o = [], 0
        for n in ns:
            st["bs"].append(ColMajor(st["x"][o:o + n].view(1, n), n, 1))
            o += n
    else:
        a, g = _matrix(case, seed)
        n = case["n"]
        st["A0"], st["A"] = a, ColMajor(torch.empty_like(a), n, n)
        st["b0"] = _entries(g, case["nrhs"], n, 0.0)
        st["x"] = ColMajor(torch.empty_like(st["b0"]), n, case["nrhs"])
    return st


def run(st):
    case, e = st["case"], st["emul"]
    if case["kind"] == "gemm":
        e.dgemm(st["A"], st["B"], st["C"], case["s"], alpha=case["alpha"], beta=case["beta"])
        return {"C": st["C"].store}
    if case["kind"] == "batched":
        st["x"].copy_(st["b0"])     # the solver overwrites the right-hand sides
        info, berr, iters = e.dgesv_batched_ir(st["As"], st["bs"])
        return {"x": st["x"], "info": info, "berr": berr, "iters": iters}
    # the factorization and the solve overwrite the matrix and the right-hand sides
    A, X = st["A"], st["x"]
    A.store.copy_(st["A0"])
    X.store.copy_(st["b0"])
    out = {"factors": A.store, "x": X.store}
    if case["kind"] == "chol":
        out["info"] = e.dpotrf(A, nb=case["nb"], slices=case["s"])
        e.dpotrs(A, X)
        return out
    if case["kind"] == "nopiv":
        ipiv, out["info"] = e.dgetrf_nopiv(A, nb=case["nb"], slices=case["s"])
    else:
        ipiv, out["info"] = e.dgetrf(A, nb=case["nb"], slices=case["s"])
    out["ipiv"] = ipiv
    e.dgetrs(A, ipiv, X)
    return out


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    """Bytes: inputs read once, outputs written once.  Operations: those of the
    kept slice-pair products, s (s + 1) / 2 for every multiply and add."""
    s = case.get("s") or 7          # the selector takes 7 on most updates
    pairs = s * (s + 1) // 2
    if case["kind"] == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 8.0 * (m * k + k * n + m * n * (2 if case["beta"] else 1)), "flops": 2.0 * m * n * k * pairs}
    if case["kind"] == "batched":
        lo, hi = case["lo"], case["hi"] + 1
        l = math.log(hi / lo)
        n2, n3 = (hi ** 2 - lo ** 2) / (2 * l), (hi ** 3 - lo ** 3) / (3 * l)   # means of n^2, n^3
        return {"bytes": 8.0 * case["count"] * n2, "flops": case["count"] * (2.0 / 3.0) * n3 * 6}   # 3 slices
    n, nrhs = case["n"], case["nrhs"]
    third = 1.0 / 3.0 if case["kind"] == "chol" else 2.0 / 3.0
    half = 0.5 if case["kind"] == "chol" else 1.0       # the lower triangle
    return {"bytes": 16.0 * (half * n * n + n * nrhs), "flops": third * n ** 3 * pairs + 2.0 * n * n * nrhs}


def exact(case, seed):
    if case["kind"] == "gemm":
        g, p = _gen(seed), case["pad"]
        m, n, k = case["m"], case["n"], case["k"]
        at, bt, ct = _entries(g, k, m + p, case["r"]), _entries(g, n, k + p, case["r"]), _entries(g, n, m + p, 0.0)
        d = bt[:, :k] @ at[:, :m]           # row j is column j of A B
        ct[:, :m] = case["alpha"] * d + (case["beta"] * ct[:, :m] if case["beta"] else 0.0)
        return {"C": ct}
    if case["kind"] == "batched":
        if case["count"] > 4096:
            return None
        ns, mats, b = _batch(case, seed)
        x, o = torch.empty_like(b), 0
        for n, m in zip(ns, mats):
            x[o:o + n] = torch.linalg.solve(m.T, b[o:o + n])
            o += n
        return {"x": x, "info": None, "berr": None, "iters": None}
    n = case["n"]
    if n > 20000:
        return None
    a, g = _matrix(case, seed)
    b = _entries(g, case["nrhs"], n, 0.0)
    out = {"info": None}
    if case["kind"] == "chol":              # symmetric: the transpose of the lower factor in the upper triangle
        l = torch.linalg.cholesky(a)
        out["factors"] = torch.tril(a, -1) + l.T
        out["x"] = torch.cholesky_solve(b.T, l).T.contiguous()
        return out
    lu, piv = torch.linalg.lu_factor(a.T, pivot=case["kind"] != "nopiv")
    out["factors"] = lu.T.contiguous()
    out["x"] = torch.linalg.lu_solve(lu, piv, b.T).T.contiguous()
    out["ipiv"] = None
    return out
