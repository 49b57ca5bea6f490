"""The calls this library is timed on: what its users have it do, through the
Python binding's public entry points, from the smallest solves to the largest.

Families
  svd      one bidiagonal, S with U and / or V^T (bdc.svd): `kind` names the
           input recipe (inputs.make), `prec` the merge products, `vectors`
           the sides formed
  values   one bidiagonal, singular values only (bdc.svd_values)
  batch    many bidiagonals of uneven sizes as one plan (bdc.BatchPlan)
  gesvd    the whole dense SVD (bdc.gesvd): square, rectangular, and tall and
           skinny (QR first)
  gebrd    the bidiagonalization alone (bdc.gebrd)

Dense inputs are Gaussian.  A batch's sizes come from its case alone, its
entries from the seed.
"""
import math

import numpy as np
import torch

from paper_2508_11467_gb300 import bdc, inputs

DEVICE = "cuda"
DTYPES = {"fp64": torch.float64, "fp32": torch.float32}


def _svd(n, kind, prec, vectors="both", **more):
    return {"family": "svd", "n": n, "kind": kind, "prec": prec, "vectors": vectors, **more}


def _values(n, kind, **more):
    return {"family": "values", "n": n, "kind": kind, **more}


def _batch(count, lo, hi, dtype, sizes, **more):
    # the leaf size and product threshold that bdc.autotune picks for such batches
    return {"family": "batch", "count": count, "lo": lo, "hi": hi, "dtype": dtype, "sizes": sizes,
            "prec": "fp64" if dtype == "fp32" else "exact", "leaf": 24 if dtype == "fp32" else 16,
            "mixed_min": 0 if dtype == "fp32" else 128, **more}


def _dense(family, m, n, **more):
    return {"family": family, "m": m, "n": n, **more}


def listed():
    return [
        # a small solve in a program's inner loop: launches and latency
        _svd(100, "uniform", "fp64", name="svd_n100_fp64"),
        # an ordinary odd-sized solve with the accurate split-BF16 products
        _svd(1001, "uniform", "exact", name="svd_n1001_exact"),
        # plain FP64, the reference precision of the method
        _svd(4096, "uniform", "fp64", name="svd_n4096_fp64"),
        # nothing deflates: every merge product at its full size
        _svd(4096, "clustered", "exact", name="svd_n4096_clustered_exact"),
        # the headline: the largest single solve
        _svd(16384, "uniform", "exact", name="svd_n16384_exact"),
        # spectra without vectors (condition numbers, ranks)
        _values(10007, "graded", name="values_n10007_graded"),
        # many small and middling problems at once, both data types
        _batch(512, 32, 1024, "fp64", 3, name="batch_512_fp64"),
        _batch(512, 32, 1024, "fp32", 3, name="batch_512_fp32"),
        # dense SVDs: small and odd, large, tall and skinny
        _dense("gesvd", 333, 333, name="gesvd_333"),
        _dense("gesvd", 4096, 4096, name="gesvd_4096"),
        _dense("gesvd", 10000, 600, name="gesvd_10000x600"),
        # the reduction alone, on a rectangular matrix
        _dense("gebrd", 1500, 1100, name="gebrd_1500x1100"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["svd", "svd", "values", "batch", "gesvd", "gesvd", "gebrd"])
    if family == "svd":
        kind = rng.choice(["uniform", "uniform", "graded", "clustered"])
        prec = rng.choice(["fp64", "exact"])
        hi = {"uniform": 16384, "graded": 16384, "clustered": 6000}[kind]
        if prec == "fp64":
            hi = 2000 if kind == "clustered" else 8192
        return _svd(_log(rng, 32, hi), kind, prec, rng.choice(["both", "both", "v", "u"]))
    if family == "values":
        kind = rng.choice(["uniform", "graded", "clustered"])
        return _values(_log(rng, 64, 4096 if kind == "clustered" else 16384), kind)
    if family == "batch":
        lo = _log(rng, 16, 128)
        return _batch(_log(rng, 32, 512), lo, _log(rng, 2 * lo, 1024), rng.choice(["fp64", "fp32"]),
                      rng.randrange(1, 1000))
    shape = rng.choice(["square", "rectangular", "tall"])
    n = _log(rng, 48, {"square": 3000, "rectangular": 2500, "tall": 1200}[shape])
    if shape == "square":
        m = n
    elif shape == "rectangular":
        m = int(n * rng.uniform(1.0, 1.5)) + 1
    else:
        m = min(_log(rng, 2 * n, 40 * n), 20000)
    return _dense(family, m, n)


def _gaussian(m, n, seed):
    g = torch.Generator(DEVICE).manual_seed(int(seed))
    return torch.randn(n, m, dtype=torch.float64, device=DEVICE, generator=g).t()


def _batch_sizes(case):
    return inputs.batch_sizes(case["count"], case["sizes"], case["lo"], case["hi"])


def _batch_entries(case, seed):
    """Diagonals and superdiagonals back to back (matrix b at offset sum(ns[:b]))."""
    total = int(_batch_sizes(case).sum())
    dt = DTYPES[case["dtype"]]
    d = torch.from_numpy(0.5 + inputs.uniform01(seed, 0, total)).to(DEVICE).to(dt)
    e = torch.from_numpy(0.5 + inputs.uniform01(seed, 1, total)).to(DEVICE).to(dt)
    return d, e


def _bidiagonal(case, seed):
    d, e = inputs.make(case["kind"], case["n"], seed)
    return torch.from_numpy(d).to(DEVICE), torch.from_numpy(e).to(DEVICE)


def prepare(case, seed):
    family = case["family"]
    if family in ("svd", "values"):
        d, e = _bidiagonal(case, seed)
        return {"case": case, "d": d, "e": e}
    if family == "batch":
        d, e = _batch_entries(case, seed)
        plan = bdc.BatchPlan(d, e, _batch_sizes(case), prec=case["prec"], leaf=case["leaf"],
                             mixed_min=case["mixed_min"], dtype=DTYPES[case["dtype"]])
        return {"case": case, "plan": plan}
    return {"case": case, "A": _gaussian(case["m"], case["n"], seed)}


def run(state):
    case = state["case"]
    family = case["family"]
    if family == "svd":
        S, U, VT, info = bdc.svd(state["d"], state["e"], prec=case["prec"], vectors=case["vectors"])
        return {"S": S, "U": U, "VT": VT, "info": info}
    if family == "values":
        S, info = bdc.svd_values(state["d"], state["e"])
        return {"S": S, "info": info}
    if family == "batch":
        plan = state["plan"]
        plan.launch()
        return {"S": plan.S, "U": plan.U, "VT": plan.VT, "info": plan.info}
    if family == "gesvd":
        S, U, VT, info = bdc.gesvd(state["A"], prec="exact")
        return {"S": S, "U": U, "VT": VT, "info": info}
    Ar, d, e, tauq, taup, info = bdc.gebrd(state["A"])
    return {"A": Ar, "d": d, "e": e, "tauq": tauq, "taup": taup, "info": info}


def work(case):
    """Inputs read and outputs written once.  Flops: the dense algorithms'
    counts; of the bidiagonal solves only the merge products of the
    clustered inputs ((8/3) n^3, (4/3) n^3 for one side): on the others
    nearly every column deflates and what is left is O(n^2) and depends on
    the data."""
    family = case["family"]
    if family in ("svd", "values"):
        n = case["n"]
        sides = 0 if family == "values" else 2 if case["vectors"] == "both" else 1
        flops = sides * 4.0 / 3.0 * n ** 3 if case["kind"] == "clustered" else 0.0
        return {"bytes": 8.0 * (3 * n - 1 + sides * n * n), "flops": flops}
    if family == "batch":
        ns = _batch_sizes(case).astype(np.float64)
        size = 4 if case["dtype"] == "fp32" else 8
        return {"bytes": size * float(np.sum(3 * ns - 1 + 2 * ns * ns)), "flops": 0.0}
    m, n = float(case["m"]), float(case["n"])
    if family == "gebrd":
        return {"bytes": 8.0 * (2 * m * n + 4 * n), "flops": 4 * m * n * n - 4 * n ** 3 / 3}
    bytes_ = 8.0 * (2 * m * n + n * n + n)
    if m >= 1.6 * n:   # QR, Q, the square SVD's reduction and back-transformations, Q U
        return {"bytes": bytes_, "flops": 2 * (2 * m * n * n - 2 * n ** 3 / 3) + 8 * n ** 3 / 3 + 4 * n ** 3
                + 2 * m * n * n}
    return {"bytes": bytes_, "flops": 4 * m * n * n - 4 * n ** 3 / 3 + (4 * m * n * n - 2 * n ** 3) + 2 * n ** 3}


# ------------------------------------------------------------- 64-bit values
def _sigma(ds, es):
    """Singular values (descending, back to back) of the upper bidiagonals
    (ds[b], es[b]): bisection on the number of singular values below a shift
    (negative pivots of B^T B - x I in stationary qd form), every value of
    every matrix at once, 15 shifts per interval."""
    points, rounds = 15, 14
    B, nmax = len(ds), max(len(d) for d in ds)
    d2 = torch.full((nmax, B), 1e200, dtype=torch.float64)
    e2 = torch.zeros((nmax, B), dtype=torch.float64)
    for b, (d, e) in enumerate(zip(ds, es)):
        d2[:len(d), b] = torch.from_numpy(d) ** 2
        e2[:len(d) - 1, b] = torch.from_numpy(e[:len(d) - 1]) ** 2
    top = [float(np.max(np.abs(d)) + (np.max(np.abs(e[:len(d) - 1])) if len(d) > 1 else 0.0)) for d, e in zip(ds, es)]
    d2, e2 = d2.to(DEVICE), e2.to(DEVICE)
    mat = torch.cat([torch.full((len(d),), b, dtype=torch.int64) for b, d in enumerate(ds)]).to(DEVICE)
    # the k-th largest of n: the point where the count of smaller ones passes n - 1 - k
    rank = torch.cat([torch.arange(len(d) - 1, -1, -1, dtype=torch.int64) for d in ds]).to(DEVICE)
    last = torch.cat([torch.full((len(d),), len(d), dtype=torch.int64) for d in ds]).to(DEVICE)
    hi = torch.tensor(top, dtype=torch.float64, device=DEVICE)[mat]
    lo = torch.zeros_like(hi)
    frac = torch.arange(1, points + 1, dtype=torch.float64, device=DEVICE)[:, None] / (points + 1)
    for _ in range(rounds):
        shift = lo + (hi - lo) * frac
        x = shift * shift
        s, count = -x, torch.zeros(x.shape, dtype=torch.int64, device=DEVICE)
        for i in range(nmax):
            a, b = (d2[i], e2[i]) if B == 1 else (d2[i][mat], e2[i][mat])
            q = a + s
            count += q < 0
            s = torch.addcmul(-x, b, s / q.masked_fill_(q == 0, 1e-300))
        below = (torch.minimum(count, last) <= rank).sum(0)      # shifts at or below the value
        width = (hi - lo) / (points + 1)
        lo, hi = lo + width * below, torch.where(below == points, hi, lo + width * (below + 1))
    return 0.5 * (lo + hi)


def _householder(x):
    """tau, beta and the vector (first entry 1) of the reflector of x."""
    alpha, tail = x[0], x[1:]
    sig2 = tail.square().sum()
    norm = torch.sqrt(alpha * alpha + sig2)
    beta = torch.where(sig2 == 0, alpha, torch.where(alpha >= 0, -norm, norm))
    tau = torch.where(sig2 == 0, torch.zeros_like(beta), (beta - alpha) / beta)
    v = torch.where(sig2 == 0, torch.zeros_like(x), x / (alpha - beta))
    v[0] = 1.0
    return tau, beta, v


def _reduce(A):
    """Unblocked bidiagonalization: (A with the reflectors, d, e, tauq, taup)."""
    A = A.contiguous().clone()
    m, n = A.shape
    d, tauq, taup = (torch.zeros(n, dtype=torch.float64, device=A.device) for _ in range(3))
    e = torch.zeros(max(n - 1, 0), dtype=torch.float64, device=A.device)
    for i in range(n):
        tauq[i], d[i], v = _householder(A[i:, i])
        T = A[i:, i + 1:]
        T -= torch.outer(tauq[i] * v, v @ T)
        A[i, i], A[i + 1:, i] = d[i], v[1:]
        if i + 1 < n:
            taup[i], e[i], u = _householder(A[i, i + 1:])
            T = A[i + 1:, i + 1:]
            T -= torch.outer(T @ u, taup[i] * u)
            A[i, i + 1], A[i, i + 2:] = e[i], u[1:]
    return A, d, e, tauq, taup


def exact(case, seed):
    """Singular values, and all of a reduction's outputs, in 64 bits by plain
    torch.  Singular vectors have no value of their own (each pair's sign is
    free)."""
    family = case["family"]
    none = {"U": None, "VT": None, "info": None}
    if family in ("svd", "values"):
        d, e = inputs.make(case["kind"], case["n"], seed)
        S = _sigma([d], [e])
        return {"S": S, "info": None} if family == "values" else {"S": S, **none}
    if family == "batch":
        d, e = (t.double().cpu().numpy() for t in _batch_entries(case, seed))
        off = np.concatenate([[0], np.cumsum(_batch_sizes(case))])
        return {"S": _sigma([d[a:b] for a, b in zip(off, off[1:])], [e[a:b] for a, b in zip(off, off[1:])]), **none}
    A, d, e, tauq, taup = _reduce(_gaussian(case["m"], case["n"], seed))
    if family == "gebrd":
        return {"A": A, "d": d, "e": e, "tauq": tauq, "taup": taup, "info": None}
    return {"S": _sigma([d.cpu().numpy()], [e.cpu().numpy()]), **none}
