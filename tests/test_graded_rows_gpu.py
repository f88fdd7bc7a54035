"""Rows of very different sizes (needs a GB300).  One-sided rotations act on each
row by itself, so the sweeps lose nothing of a small row: the singular values
of D B, D diagonal and B well conditioned, come out to a relative error of
about n u cond(B), however small."""
import numpy as np
import pytest
import torch

import __graft_entry__  # noqa: F401
import oracle
import paper_2601_17979_gb300 as bsvd
from oracle import checks

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()


def row_graded(rng, m, n, span, dtype):
    """D B and cond(B), D from 1 to 2^-span in any order."""
    B = rng.standard_normal((m, n)) + (1j * rng.standard_normal((m, n)) if np.issubdtype(dtype, np.complexfloating) else 0)
    d = 2.0 ** -rng.permutation(np.linspace(0, span, m).round())
    return (B * d[:, None]).astype(dtype), np.linalg.cond(B)


def relative_errors(mats, **kw):
    wide = [x.astype(np.complex128 if np.iscomplexobj(x) else np.float64) for x in mats]
    ref = oracle.gesvj(wide)["S"]
    r = bsvd.gesvj(torch.from_numpy(np.stack(mats)).cuda(), **kw)
    torch.cuda.synchronize()
    assert int(r.info.max()) == 0
    S = r.S.cpu().numpy().astype(np.float64)
    return np.array([(np.abs(S[k] - ref[k]) / ref[k]).max() for k in range(len(mats))])


# The factorisations of the preconditioned start are accurate relative to each
# column only.  Against the plain start (inner_sweeps = 1) of the same call:
# both within their scatter, a factor of three, and one rounding per column.
@pytest.mark.parametrize("dtype", [np.float32, np.float64, np.complex64, np.complex128])
@pytest.mark.parametrize("span", [6, 8, 10])
@pytest.mark.parametrize("n,nb", [(40, 8), (40, 16), (64, 16)])
def test_preconditioned_start_keeps_small_values(n, nb, span, dtype):
    rng = np.random.default_rng(n + span)
    mats = [row_graded(rng, n, n, span, dtype)[0] for _ in range(24)]
    err, plain = relative_errors(mats, nb=nb), relative_errors(mats, nb=nb, inner_sweeps=1)
    assert np.median(err) <= 3 * np.median(plain) + n * checks.unit_roundoff(dtype), (np.median(err), np.median(plain))


# The mixed path's restoration of V, whose small entries count where the columns
# are graded too: within ten times the FP64 pipe's error on the same matrices
# (complex128 restores V there).
@pytest.mark.parametrize("n", [40, 96])
def test_mixed_graded_rows_and_columns(n):
    rng = np.random.default_rng(n)
    mats = []
    for _ in range(12):
        A = row_graded(rng, n, n, 60, np.float64)[0]
        mats.append(A * 2.0 ** -rng.permutation(np.linspace(0, 60, n).round()))
    err = relative_errors(mats, prec="mixed")
    cplx = relative_errors([x.astype(np.complex128) for x in mats], prec="mixed")
    assert np.median(err) <= 10 * np.median(cplx), (np.median(err), np.median(cplx))


# Gram blocks and updates as digit products (nb = 8, 16) are left out for such
# matrices, on chip, in global slots and on the multi-kernel path; one row more
# than the limit of 2^6 spans, and far beyond it.  Wide matrices: graded columns.
@pytest.mark.parametrize("dtype", [np.float64, np.complex128])
@pytest.mark.parametrize("nb", [8, 16])
@pytest.mark.parametrize("path", ["fused", "blocked", "slots"])
@pytest.mark.parametrize("m,n", [(24, 24), (40, 40), (57, 33), (33, 70)])
def test_small_values_of_graded_rows(m, n, path, nb, dtype):
    rng = np.random.default_rng(m + n)
    u = checks.unit_roundoff(dtype)
    mats, cond = [], []
    for span in (7, 8, 20, 40, 60, 100):
        A, c = row_graded(rng, max(m, n), min(m, n), span, dtype)
        mats.append(A if m >= n else np.ascontiguousarray(A.conj().T))
        cond.append(c)
    T = [torch.from_numpy(np.asfortranarray(x)).cuda() for x in mats]
    if path == "slots":
        r = bsvd.gesvj_batched(T, path="persistent", nb=nb, flags=bsvd.FLAG_NO_ONCHIP)
    else:
        r = bsvd.gesvj_batched(T, path=path, nb=nb)
    torch.cuda.synchronize()
    ref = oracle.gesvj(mats)["S"]
    for k, A in enumerate(mats):
        S = r.S[k].cpu().numpy()
        rel = (np.abs(S - ref[k]) / ref[k]).max()
        assert int(r.info[k]) == 0 and rel <= 50 * min(m, n) * u * cond[k], (k, int(r.info[k]), rel / u, cond[k])


def kahan(m, n, theta=1.2):
    s, c = np.sin(theta), np.cos(theta)
    return (s ** np.arange(m))[:, None] * (np.eye(m, n) - c * np.triu(np.ones((m, n)), 1))


# Cross-only sweeps take more of them on such matrices (Kahan's 200 x 140: 16
# against 10), so these run the sweeps of inner_sweeps = 1: the same bits.
@pytest.mark.parametrize("dtype", [np.float64, np.complex128])
@pytest.mark.parametrize("path", ["auto", "blocked", "slots"])
@pytest.mark.parametrize("m,n", [(64, 64), (96, 70), (200, 140)])
def test_graded_rows_take_full_sweeps(m, n, path, dtype):
    rng = np.random.default_rng(m)
    mats = [kahan(m, n).astype(dtype), row_graded(rng, m, n, 30, dtype)[0]]
    T = [torch.from_numpy(np.asfortranarray(x)).cuda() for x in mats]
    kw = dict(path="persistent", flags=bsvd.FLAG_NO_ONCHIP) if path == "slots" else dict(path=path)
    r, f = bsvd.gesvj_batched(T, **kw), bsvd.gesvj_batched(T, inner_sweeps=1, **kw)
    torch.cuda.synchronize()
    for k in range(len(mats)):
        assert int(r.info[k]) == 0 and int(r.sweeps[k]) == int(f.sweeps[k]), (k, int(r.sweeps[k]), int(f.sweeps[k]))
        assert torch.equal(r.S[k], f.S[k]) and torch.equal(r.U[k], f.U[k]) and torch.equal(r.V[k], f.V[k])


# Tall matrices whose rows span seven orders keep the preconditioned start (and,
# in FP64, the digit products): fewer sweeps than the plain start, no larger error.
# (Sizes on chip: the multi-kernel path has no such start.)
@pytest.mark.parametrize("dtype,m,n", [(np.float32, 128, 64), (np.float64, 128, 64), (np.float64, 100, 48),
                                       (np.complex64, 100, 48), (np.complex128, 80, 36)])
def test_tall_matrices_of_seven_orders_keep_the_start(m, n, dtype):
    rng = np.random.default_rng(m)
    mats = []
    while len(mats) < 16:
        A = row_graded(rng, m, n, 4, np.complex128 if np.issubdtype(dtype, np.complexfloating) else np.float64)[0]
        A *= 10.0 ** -np.linspace(0, 2, n)                   # not a flat spectrum
        e = np.frexp(np.abs(A).max(1))[1]
        A[e.argmin()] *= 2.0 ** (e.max() - 7 - e.min())
        mats.append(A.astype(dtype))
    err, plain = relative_errors(mats, nb=16), relative_errors(mats, nb=16, inner_sweeps=1)
    assert np.median(err) <= 3 * np.median(plain) + n * checks.unit_roundoff(dtype), (np.median(err), np.median(plain))
    A = torch.from_numpy(np.stack(mats)).cuda()
    sweeps, full = int(bsvd.gesvj(A, nb=16).sweeps.sum()), int(bsvd.gesvj(A, nb=16, inner_sweeps=1).sweeps.sum())
    assert sweeps < full, (sweeps, full)


# The mixed path keeps only V of its single-precision solve, which may start
# preconditioned up to ten orders: the values are the FP64 sweeps' all the same.
@pytest.mark.parametrize("dtype", [np.float64, np.complex128])
@pytest.mark.parametrize("span", [5, 7, 9])
@pytest.mark.parametrize("n", [40, 64, 96])
def test_mixed_values_of_moderately_graded_rows(n, span, dtype):
    rng = np.random.default_rng(n + span)
    mats = [row_graded(rng, n, n, span, dtype)[0] for _ in range(16)]
    err, plain = relative_errors(mats, prec="mixed"), relative_errors(mats, inner_sweeps=1)
    assert np.median(err) <= 3 * np.median(plain) + n * checks.unit_roundoff(dtype), (np.median(err), np.median(plain))
