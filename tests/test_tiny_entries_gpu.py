"""Entries near the bottom of the type's range beside entries of size one
(needs a GB300): a reflection whose first entry is denormal, in the QR and in
the LQ.  Bounds as in test_parity_gpu."""
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


@pytest.mark.parametrize("dtype", [np.float32, np.float64, np.complex64, np.complex128])
@pytest.mark.parametrize("m,n,nb", [(64, 64, 16), (97, 45, 16), (90, 40, 8), (300, 20, 16), (45, 97, 16)])
@pytest.mark.parametrize("path", ["auto", "persistent"])
def test_denormal_entries(path, m, n, nb, dtype):
    rng = np.random.default_rng(m + n)
    cplx = np.issubdtype(dtype, np.complexfloating)
    tiny = [1e-41, 1e-44, 1e-38] if dtype in (np.float32, np.complex64) else [1e-310, 5e-324, 1e-307]
    mats = []
    for t in tiny:
        for rows in ([0], [0, m // 2], list(range(0, m, 2))):
            A = rng.standard_normal((m, n)) + (1j * rng.standard_normal((m, n)) if cplx else 0)
            for r in rows:                                   # some of the row's entries: no row is small
                A[r, rng.random(n) < 0.6] = t
            mats.append(A.astype(dtype))
    r = bsvd.gesvj_batched([torch.from_numpy(np.asfortranarray(x)).cuda() for x in mats], path=path, nb=nb)
    torch.cuda.synchronize()
    u = checks.unit_roundoff(dtype)
    wide = [x.astype(np.complex128 if cplx else np.float64) for x in mats]
    ref = oracle.gesvj(wide)["S"]
    for i, A in enumerate(wide):
        assert int(r.info[i]) == 0, i
        meas = checks.measures(A, r.S[i].cpu().numpy(), r.U[i].cpu().numpy(), r.V[i].cpu().numpy(), ref[i])
        assert checks.violations(meas, u) == [], (i, meas)


@pytest.mark.parametrize("dtype,low", [(np.complex64, 62), (np.complex128, 508)])
@pytest.mark.parametrize("m,n,nb", [(60, 48, 16), (30, 24, 8), (40, 40, 4), (90, 40, 16)])
@pytest.mark.parametrize("path", ["auto", "blocked"])
def test_rotations_of_denormal_gram_entries(path, m, n, nb, dtype, low):
    """Short columns whose Gram entries are near the bottom of the range or
    denormal: the rotations stay unitary, so V and the product keep their
    bounds (U's columns then have no accurate Gram entries to go by)."""
    rng = np.random.default_rng(m)
    u = checks.unit_roundoff(dtype)
    mats = []
    for k in (low, low + 4, low + 8, low + 12):
        A = rng.standard_normal((m, n)) + 1j * rng.standard_normal((m, n))
        A[:, n // 2:] *= 2.0 ** -k
        mats.append(A.astype(dtype))
        mats.append((A.conj() * 2.0 ** -np.linspace(0, 3, n).round()).astype(dtype))
    r = bsvd.gesvj_batched([torch.from_numpy(np.asfortranarray(x)).cuda() for x in mats], path=path, nb=nb)
    torch.cuda.synchronize()
    for i, A in enumerate(mats):
        meas = checks.measures(A.astype(np.complex128), r.S[i].cpu().numpy(), r.U[i].cpu().numpy(), r.V[i].cpu().numpy())
        assert not {"resid", "orth_v"} & set(checks.violations(meas, u)), (i, meas)


@pytest.mark.parametrize("dtype", [np.float64, np.complex128])
@pytest.mark.parametrize("m,n,nb", [(48, 32, 16), (70, 48, 16), (64, 64, 16), (30, 16, 8), (40, 40, 8)])
@pytest.mark.parametrize("path", ["auto", "blocked", "slots", "mixed"])
def test_columns_short_of_the_squares(path, m, n, nb, dtype):
    """Dense columns of 2^-520, 2^-560 and 2^-600 (their squares underflow) in one
    block pair with columns of size one: as on the FP64 pipe (nb = 4), which
    orthogonalises the first and leaves the others as they are."""
    rng = np.random.default_rng(m + n)
    mats = []
    for at in ([0, 1, 2], [n - 1, n // 2, 3], [n - 3, n - 2, n - 1]):
        A = rng.standard_normal((m, n)) + (1j * rng.standard_normal((m, n)) if dtype == np.complex128 else 0)
        A[:, at] *= 2.0 ** -np.array([520, 560, 600])
        mats.append(A.astype(dtype))
    T = [torch.from_numpy(np.asfortranarray(x)).cuda() for x in mats]

    def call(nb):
        if path == "slots":
            return bsvd.gesvj_batched(T, path="persistent", nb=nb, flags=bsvd.FLAG_NO_ONCHIP)
        return bsvd.gesvj_batched(T, prec="mixed", nb=nb) if path == "mixed" else bsvd.gesvj_batched(T, path=path, nb=nb)
    r, p = call(nb), call(4)
    torch.cuda.synchronize()
    # a pair is rotated to 30 u of orthogonal, so S differs by less than n 30 u of itself; doubled
    tol = 2 * 30 * n * checks.U64
    for k, A in enumerate(mats):
        S, P = r.S[k].cpu().numpy(), p.S[k].cpu().numpy()
        assert int(r.info[k]) == 0 and int(p.info[k]) == 0
        rel = np.abs(S - P) / P
        assert rel[-3:].max() <= tol, (k, S[-3:], P[-3:])
        meas = checks.measures(A, S, r.U[k].cpu().numpy(), r.V[k].cpu().numpy(), P)
        assert not {"sigma_err", "resid", "orth_v"} & set(checks.violations(meas, checks.U64)), (k, meas)
