"""Workloads of the batched SVD as a user's program runs them: what is timed
and compared when a kernel changes.

A case is one batch of matrices and the options of the call.  One pass makes
the call and multiplies the factors back: with U diag(S) V^H and the
Gram matrices U^H U and V^H V, a program checks or uses an SVD without
depending on what the decomposition leaves open (the sign or phase of each
vector pair, the basis inside a cluster of equal singular values), and
these, S and info are the outputs.  Calls that ask for no vectors return S
and info.  The sweep counts are a diagnostic of the iteration and are not
part of the result.

Sizes and distributions are those of this repository's benchmark and tests:
the 32 x 32, 128 x 64 and clustered 96 x 96 batches, the uneven batch, the
squares and the tall-skinny panels of the paper's figures.  The serving loop
is left out: what it batches together depends on arrival times, and it runs
the kernels of the batch calls below.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2601_17979_gb300 as bsvd

DTYPES = {"f32": torch.float32, "f64": torch.float64, "c64": torch.complex64, "c128": torch.complex128}
WIDE = {"f32": torch.float64, "f64": torch.float64, "c64": torch.complex128, "c128": torch.complex128}
UNEVEN_SHAPES = 24          # distinct shapes of an uneven batch


def listed():
    def case(name, dtype, batch, m, n, dist, **options):
        d = {"name": name, "kind": "strided", "dtype": dtype, "batch": batch, "m": m, "n": n, "dist": dist,
             "vectors": True, "prec": "native", "qr": False, "nb": 0, "tol_u": 0.0}
        d.update(options)
        return d

    return [
        # one small matrix: the latency of a call
        case("one_64x64_f32", "f32", 1, 64, 64, "normal"),
        # the paper-style batch of very small matrices, with its own block width and tolerance
        case("square32_f64", "f64", 1000, 32, 32, "normal", nb=8, tol_u=32.0),
        # the headline batch: tall matrices with a geometric spectrum, double and single precision
        case("tall128x64_f64", "f64", 4000, 128, 64, "geo1e6", nb=16),
        case("tall128x64_f32", "f32", 10000, 128, 64, "geo1e3", nb=16),
        # FP64 results from mostly FP32 work, clustered spectrum of condition number 1e8
        case("mixed96_f64", "f64", 2000, 96, 96, "clustered", prec="mixed", nb=16),
        # a ragged size in complex double precision, every option left to the library
        case("ragged75x50_c128", "c128", 500, 75, 50, "normal"),
        # wide matrices, singular values only
        case("wide45x97_values_c64", "c64", 3000, 45, 97, "normal", vectors=False),
        # tall-skinny panels
        case("panel1000x16_f64", "f64", 1000, 1000, 16, "uniform01"),
        # the paper's squares, too large for one SM's shared memory, in three types
        case("square512_f32", "f32", 128, 512, 512, "uniform01"),
        case("square256_c64", "c64", 200, 256, 256, "uniform01"),
        case("square256_f64", "f64", 64, 256, 256, "uniform01"),
        # an uneven batch (sizes from 8 to 512) in one pointer-array call
        {"name": "uneven_f32", "kind": "uneven", "dtype": "f32", "per_shape": 60, "shape_seed": 4, "lo": 8, "hi": 512,
         "vectors": True},
    ]


def _cost(dtype, batch, m, n):
    """Rough cost of a batch, in units of one FP64 multiply-add chain: for bounding drawn cases."""
    w = {"f32": 1 / 12, "f64": 1.0, "c64": 1 / 8, "c128": 4.0}[dtype]
    return w * batch * max(m, n) * min(m, n) ** 2


_COST_MAX = 1.2e9


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    dtype = rng.choice(["f32", "f32", "f64", "f64", "c64", "c128"])
    if rng.random() < 0.15 and dtype in ("f32", "c64"):
        return {"kind": "uneven", "dtype": dtype, "per_shape": _log(rng, 4, 40), "shape_seed": rng.randrange(1, 10 ** 6),
                "lo": 8, "hi": _log(rng, 64, 400), "vectors": rng.random() < 0.8}
    big = _log(rng, 8, 512)
    form = rng.random()
    if form < 0.35:
        m, n = big, big
    elif form < 0.55:
        m, n = big, (big + 1) // 2
    elif form < 0.7:
        m, n = _log(rng, 200, 2000), rng.randint(5, 24)
    else:
        m, n = big, rng.randint(max(4, big // 5), big)
    if dtype == "c128" and m * n * n > 6e6:          # the costliest type: up to about 180 x 180
        m, n = min(m, 180), min(n, 150)
    tall = m >= 8 * n
    if rng.random() < 0.2:
        m, n = n, m
    cap = max(1, min(10000, int(_COST_MAX / max(_cost(dtype, 1, m, n), 1.0)), int(3e8 / (m * n * 16))))
    batch = _log(rng, 1, cap)
    prec = "mixed" if dtype in ("f64", "c128") and rng.random() < 0.25 else "native"
    # graded spectra come with the small and medium sizes, as in the benchmark; the large ones are U[0, 1] or normal
    dists = ["normal", "uniform01", "geo1e3"] if min(m, n) <= 128 else ["normal", "uniform01"]
    return {"kind": "strided", "dtype": dtype, "batch": batch, "m": m, "n": n,
            "dist": rng.choice(dists), "vectors": rng.random() < 0.85, "prec": prec,
            "qr": bool(tall and prec == "native" and rng.random() < 0.4), "nb": 0, "tol_u": 0.0}


# ---- inputs ---------------------------------------------------------------

def _normal(g, shape, cplx):
    if cplx:
        return torch.complex(torch.randn(shape, generator=g, device="cuda", dtype=torch.float64),
                             torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)) / math.sqrt(2.0)
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)


def _uniform(g, shape, cplx, lo, hi):
    x = lo + (hi - lo) * torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)
    if cplx:
        x = torch.complex(x, lo + (hi - lo) * torch.rand(shape, generator=g, device="cuda", dtype=torch.float64))
    return x


def _haar_small(g, shape, cplx):
    """Matrices with orthonormal columns: 16 random reflections applied to the leading columns of I, in one product
    per side (quick to make; Haar enough to mix every row and column)."""
    b, r, c = shape
    dt = torch.complex128 if cplx else torch.float64
    X = torch.eye(r, c, dtype=dt, device="cuda").expand(b, r, c).clone()
    for _ in range(16):
        v = _normal(g, (b, r, 1), cplx)
        v /= torch.linalg.vector_norm(v, dim=1, keepdim=True)
        X -= 2 * v @ (v.mH @ X)
    return X


def _spectrum(dist, k):
    i = torch.arange(k, dtype=torch.float64, device="cuda")
    if dist == "geo1e6":
        return 10.0 ** (-6.0 * i / max(k - 1, 1))
    if dist == "geo1e3":
        return 10.0 ** (-3.0 * i / max(k - 1, 1))
    if dist == "clustered":                       # pairs (c, c (1 - 1e-6)), c from 1 to 1e-8
        c = 10.0 ** (-8.0 * (i // 2) / max((k + 1) // 2 - 1, 1))
        return c * (1.0 - 1e-6 * (i % 2))
    raise ValueError(dist)


def _matrices(g, dist, b, m, n, dtype):
    cplx = dtype in ("c64", "c128")
    if dist == "normal":
        A = _normal(g, (b, m, n), cplx)
    elif dist == "uniform01":
        A = _uniform(g, (b, m, n), cplx, 0.0, 1.0)
    elif dist == "uniform11":
        A = _uniform(g, (b, m, n), cplx, -1.0, 1.0)
    else:
        k = min(m, n)
        A = (_haar_small(g, (b, m, k), cplx) * _spectrum(dist, k)) @ _haar_small(g, (b, n, k), cplx).mH
    A = A.to(DTYPES[dtype])
    return A.transpose(1, 2).contiguous().transpose(1, 2)      # column-major matrices, as LAPACK stores them


def _shapes(case):
    r = np.random.default_rng(case["shape_seed"])
    out = []
    for _ in range(UNEVEN_SHAPES):
        m = int(r.integers(case["lo"], case["hi"] + 1))
        out.append((m, int(r.integers(case["lo"], m + 1))))
    return out


def _inputs(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if case["kind"] == "uneven":
        return [_matrices(g, "uniform11", case["per_shape"], m, n, case["dtype"]) for m, n in _shapes(case)]
    return _matrices(g, case["dist"], case["batch"], case["m"], case["n"], case["dtype"])


def prepare(case, seed):
    A = _inputs(case, seed)
    st = {"case": case, "A": A}
    if case["kind"] == "uneven":
        st["mats"] = [X[i] for X in A for i in range(X.shape[0])]
    else:
        u = 2.0 ** -53 if case["dtype"] in ("f64", "c128") else 2.0 ** -24
        st["opts"] = {"nb": case["nb"], "tol": case["tol_u"] * u, "prec": case["prec"],
                      "flags": bsvd.FLAG_QR if case["qr"] else 0}
    return st


# ---- one pass ---------------------------------------------------------------

def _products(S, U, V):
    return (U * S.unsqueeze(-2)) @ V.mH, U.mH @ U, V.mH @ V


def run(state):
    case = state["case"]
    vectors = case["vectors"]
    if case["kind"] == "uneven":
        r = bsvd.gesvj_batched(state["mats"], compute_u=vectors, compute_v=vectors, path="persistent",
                               flags=bsvd.FLAG_SPLIT_LARGE | bsvd.FLAG_SPLIT_F32)
        out = {"S": torch.cat(r.S), "info": r.info}
        if vectors:
            p = case["per_shape"]
            parts = [_products(torch.stack(r.S[i:i + p]), torch.stack(r.U[i:i + p]), torch.stack(r.V[i:i + p]))
                     for i in range(0, len(r.S), p)]
            for key, xs in zip(("A", "UU", "VV"), zip(*parts)):
                out[key] = torch.cat([x.reshape(-1) for x in xs])
        return out
    r = bsvd.gesvj(state["A"], compute_u=vectors, compute_v=vectors, **state["opts"])
    out = {"S": r.S, "info": r.info}
    if vectors:
        out["A"], out["UU"], out["VV"] = _products(r.S, r.U, r.V)
    return out


# ---- what a pass cannot do without ------------------------------------------

def work(case):
    """Bytes: the matrices in, S, U and V out.  Operations: the direct (R-bidiagonalisation) count for the thin SVD,
    6 m n^2 + 11 n^3 with the vectors and 2 m n^2 + 2 n^3 without; four times that for complex data."""
    elt = {"f32": 4, "f64": 8, "c64": 8, "c128": 16}[case["dtype"]]
    cplx = 4 if case["dtype"] in ("c64", "c128") else 1
    shapes = [(m, n, case["per_shape"]) for m, n in _shapes(case)] if case["kind"] == "uneven" else \
        [(case["m"], case["n"], case["batch"])]
    nbytes = flops = 0.0
    for m, n, b in shapes:
        M, N = max(m, n), min(m, n)
        nbytes += b * (M * N + N) * elt
        if case["vectors"]:
            nbytes += b * (M * N + N * N) * elt
            flops += b * cplx * (6 * M * N * N + 11 * N ** 3)
        else:
            flops += b * cplx * (2 * M * N * N + 2 * N ** 3)
    return {"bytes": nbytes, "flops": flops}


# ---- the same outputs in 64 bits ----------------------------------------------

def exact(case, seed):
    """The singular values by LAPACK in 64 bits; the product is the matrix itself, the Gram matrices are I."""
    A = _inputs(case, seed)
    groups = A if case["kind"] == "uneven" else [A]
    vectors = case["vectors"]
    S, P, G = [], [], []
    for X in groups:
        X = X.to(WIDE[case["dtype"]]).cpu()
        S.append(torch.from_numpy(np.linalg.svd(X.numpy(), compute_uv=False)))
        if vectors:
            k = S[-1].shape[1]
            P.append(X)
            G.append(torch.eye(k, dtype=X.dtype).expand(X.shape[0], k, k))
    out = {"S": S[0], "info": None}
    if case["kind"] == "uneven":
        out["S"] = torch.cat([s.reshape(-1) for s in S])
    if vectors:
        cat = (lambda xs: torch.cat([x.reshape(-1) for x in xs])) if case["kind"] == "uneven" else (lambda xs: xs[0])
        out["A"], out["UU"], out["VV"] = cat(P), cat(G), cat(G)
    return out
