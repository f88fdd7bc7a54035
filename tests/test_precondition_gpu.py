"""The preconditioned start of the on-chip and persistent solvers (needs a
GB300): a pivoted QR, an LQ, the sweeps on the triangular factor, the left
vectors through Q.  Bounds as in test_parity_gpu, against the oracle, and the
singular values against the plain start (inner_sweeps = 1) of the same call."""
import numpy as np
import pytest
import torch

import __graft_entry__  # noqa: F401
import oracle
import paper_2601_17979_gb300 as bsvd
import synth
from oracle import checks

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()


def run(mats, **kw):
    r = bsvd.gesvj(torch.from_numpy(np.stack(mats)).cuda(), **kw)
    torch.cuda.synchronize()
    return [None if x is None else x.cpu().numpy() for x in (r.S, r.U, r.V, r.info)]


def check(mats, S, U, V, info, label):
    ref = oracle.gesvj(mats)["S"]
    u = checks.unit_roundoff(mats[0].dtype)
    for i, A in enumerate(mats):
        assert info[i] == 0, (label, i)
        meas = checks.measures(A, S[i], None if U is None else U[i], None if V is None else V[i], ref[i])
        assert checks.violations(meas, u) == [], (label, i, meas)


def graded(rng, m, n, dtype, kappa=1e4):
    cplx = np.issubdtype(dtype, np.complexfloating)
    return synth.with_sigma(rng, m, n, synth.sigma_family("geo", min(m, n), kappa), cplx).astype(dtype)


# nb = 16 and 8; one block column more and less than a full block; M = N, M just
# above N, M >= 8 N; odd block counts; the widest that fit; wide matrices
SHAPES = [(33, 33, 16), (47, 33, 16), (48, 48, 16), (49, 49, 16), (64, 64, 16), (97, 65, 16), (128, 64, 16), (65, 128, 16),
          (100, 81, 16), (300, 20, 16), (17, 17, 8), (47, 47, 8), (46, 35, 8), (23, 40, 8), (160, 16, 8), (400, 5, 8),
          (700, 9, 8)]


@pytest.mark.parametrize("dtype", [np.float32, np.float64, np.complex64, np.complex128])
@pytest.mark.parametrize("m,n,nb", SHAPES)
def test_preconditioned_shapes(dtype, m, n, nb):
    rng = np.random.default_rng(m * 131 + n + nb)
    cplx = np.issubdtype(dtype, np.complexfloating)
    mats = [graded(rng, m, n, dtype, 1e3 if dtype in (np.float32, np.complex64) else 1e6) for _ in range(3)]
    mats.append((rng.standard_normal((m, n)) + (1j * rng.standard_normal((m, n)) if cplx else 0)).astype(dtype))
    S, U, V, info = run(mats, nb=nb)
    check(mats, S, U, V, info, f"{dtype.__name__} {m}x{n}")
    S1 = run(mats, nb=nb, inner_sweeps=1)[0]
    u = checks.unit_roundoff(dtype)
    assert np.abs(S - S1).max() <= 2 * 50 * min(m, n) * u * S1.max()
    S2, U2, V2, info2 = run(mats, nb=nb, compute_u=False)
    check(mats, S2, None, V2, info2, "jobu=N")
    S3, U3, V3, info3 = run(mats, nb=nb, compute_v=False)
    check(mats, S3, U3, None, info3, "jobv=N")


@pytest.mark.parametrize("dtype", [np.float32, np.float64, np.complex64, np.complex128])
@pytest.mark.parametrize("n", [40, 64])
def test_deficient_and_extreme_columns(dtype, n):
    """A zero column (the plain start), equal columns, a rank of 5, columns
    scaled down to 2^-60 and the identity."""
    rng = np.random.default_rng(n)
    cplx = np.issubdtype(dtype, np.complexfloating)

    def rand(*s):
        return rng.standard_normal(s) + (1j * rng.standard_normal(s) if cplx else 0)
    Z = rand(n + 9, n)
    Z[:, 3] = 0
    E = rand(n + 9, n)
    E[:, n - 1] = E[:, 0]
    E[:, 7] = E[:, 0]
    Rk = rand(n + 9, 5) @ rand(5, n)
    G = rand(n + 9, n) * 2.0 ** -np.linspace(0, 60, n).round()
    mats = [x.astype(dtype) for x in (Z, E, Rk, G, np.eye(n + 9, n) + 0 * Z)]
    for nb in (8, 16):
        S, U, V, info = run(mats, nb=nb)
        check(mats, S, U, V, info, f"nb {nb}")


@pytest.mark.parametrize("dtype", [np.float32, np.float64, np.complex128])
def test_small_singular_values_of_scaled_columns(dtype):
    """A = B D with B well conditioned: one-sided Jacobi finds every singular
    value to a relative error of about n u cond(B), however D grades (and in any
    order); the factorisations keep that."""
    rng = np.random.default_rng(9)
    n, m = 64, 80
    d = 2.0 ** -rng.permutation(np.linspace(0, 30, n).round())
    mats, cond = [], []
    for _ in range(3):
        B = rng.standard_normal((m, n)) + (1j * rng.standard_normal((m, n)) if dtype == np.complex128 else 0)
        mats.append((B * d).astype(dtype))
        cond.append(np.linalg.cond(B / np.linalg.norm(B, axis=0)))
    S = run(mats, nb=16)[0]
    ref = oracle.gesvj(mats)["S"]
    u = checks.unit_roundoff(dtype)
    for k in range(3):
        rel = np.abs(S[k] - ref[k]) / ref[k]
        assert rel.max() <= 50 * n * u * cond[k], (k, rel.max())


@pytest.mark.parametrize("dtype", [np.float32, np.float64, np.complex64, np.complex128])
def test_small_singular_values_of_scaled_rows(dtype):
    """Rows of very different sizes: the plain start is kept, and with it the
    small singular values' relative accuracy."""
    rng = np.random.default_rng(10)
    m, n = 70, 48
    B = rng.standard_normal((m, n)) + (1j * rng.standard_normal((m, n)) if np.issubdtype(dtype, np.complexfloating) else 0)
    B[::3] *= 2.0 ** -40                                     # 46 rows of size 1: two singular values near 2^-40
    mats = [B.astype(dtype)]
    ref = oracle.gesvj(mats)["S"][0]
    assert ref[-3] > 1e-3 and ref[-2] < 1e-10
    S = run(mats, nb=16)[0][0]
    cond = np.linalg.cond(B[np.arange(m) % 3 != 0])
    assert np.abs(S - ref)[-2:].max() <= 50 * n * checks.unit_roundoff(dtype) * cond * ref[-2]


@pytest.mark.parametrize("m,n", [(128, 64), (96, 96), (64, 100), (33, 20), (9, 3)])
@pytest.mark.parametrize("dtype", [np.float64, np.complex128])
def test_mixed_restoration(m, n, dtype):
    """Graded and clustered spectra through the preconditioned restoration of
    the mixed path, at the scale 1 and scaled by 2^500 (where it is skipped)."""
    rng = np.random.default_rng(m + n)
    cplx = dtype == np.complex128
    k = min(m, n)
    mats = [graded(rng, m, n, dtype, 1e6), synth.with_sigma(rng, m, n, synth.clustered_pairs(k), cplx),
            np.ldexp(1.0, 500) * graded(rng, m, n, dtype, 1e6)]
    S, U, V, info = run(mats, prec="mixed")
    assert (info == 0).all()
    S[2], mats[2] = S[2] * 2.0 ** -500, mats[2] * 2.0 ** -500
    check(mats, S, U, V, info, "mixed")


# fewer columns than the CTA has warps: reductions share the scratch with the
# norms and the permutation
@pytest.mark.parametrize("dtype", [np.float32, np.float64, np.complex64, np.complex128])
@pytest.mark.parametrize("m,n", [(1, 1), (40, 1), (1, 9), (40, 2), (2, 2), (40, 3), (3, 60), (90, 7)])
def test_few_columns(m, n, dtype):
    rng = np.random.default_rng(31 * m + n)
    cplx = np.issubdtype(dtype, np.complexfloating)
    mats = [(rng.standard_normal((m, n)) + (1j * rng.standard_normal((m, n)) if cplx else 0)).astype(dtype) for _ in range(3)]
    for kw in [dict(nb=8), dict(nb=16)] + ([dict(nb=16, prec="mixed")] if dtype in (np.float64, np.complex128) else []):
        S, U, V, info = run(mats, **kw)
        check(mats, S, U, V, info, f"{dtype.__name__} {m}x{n} {kw}")
