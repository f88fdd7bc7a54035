"""FP64 and complex128 Gram blocks and updates as exact digit products on the
tensor cores (nb = 8, 16; needs a GB300): on chip, multi-kernel, persistent in global slots.
Bounds as in test_parity_gpu against the oracle."""
import numpy as np
import pytest
import torch

import __graft_entry__  # noqa: F401
import oracle
import paper_2601_17979_gb300 as bsvd
from oracle import checks

pytestmark = pytest.mark.gpu
U = checks.U64


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()


def normal(rng, shape, cplx=False):
    x = rng.standard_normal(shape)
    return x + 1j * rng.standard_normal(shape) if cplx else x


def run(mats, path, nb=16, **kw):
    T = [torch.from_numpy(np.ascontiguousarray(x.T)).cuda().t() for x in mats]
    if path == "slots":
        r = bsvd.gesvj_batched(T, path="persistent", nb=nb, flags=bsvd.FLAG_NO_ONCHIP, **kw)
    else:
        r = bsvd.gesvj_batched(T, path=path, nb=nb, **kw)
    torch.cuda.synchronize()
    return ([x.cpu().numpy() for x in r.S], [x.cpu().numpy() for x in r.U], [x.cpu().numpy() for x in r.V],
            r.info.cpu().numpy())


def check(mats, out, label):
    S, Uo, V, info = out
    ref = oracle.gesvj(mats)["S"]
    for i, A in enumerate(mats):
        assert info[i] == 0, (label, i)
        meas = checks.measures(A, S[i], Uo[i], V[i], ref[i])
        assert checks.violations(meas, U) == [], (label, i, A.shape, meas)


# rows one more and less than the 16-row tiles and than the four warps' 64, a
# single tile, few columns beside a full block, odd block counts
SHAPES = [(17, 17), (31, 20), (48, 33), (63, 47), (64, 64), (65, 49), (81, 80), (127, 40), (40, 90)]


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("nb", [8, 16])
@pytest.mark.parametrize("path", ["fused", "blocked", "slots"])
def test_shapes(path, nb, cplx):
    rng = np.random.default_rng(5)
    shapes = SHAPES if not (cplx and path == "fused") else [s for s in SHAPES if max(s) * min(s) < 3500]   # fits on chip
    mats = [normal(rng, s, cplx) for s in shapes]
    check(mats, run(mats, path, nb), path)


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("path", ["fused", "blocked", "slots"])
def test_exponent_ranges(path, cplx):
    """Rows and columns scaled over hundreds of binary orders, tiny and zero
    entries, equal magnitudes, and blocks in which J = I is applied (no masks)."""
    rng = np.random.default_rng(6)
    n = 48
    B = normal(rng, (70, n), cplx)
    # (over 2^200 complex128 runs into the sweep limit on the FP64 pipe as well)
    rows = B * 2.0 ** -np.linspace(0, 100 if cplx else 300, 70).round()[:, None]
    cols = B * 2.0 ** -np.linspace(0, 60, n).round()
    both = rows * 2.0 ** -np.linspace(0, 60, n).round()
    sparse = B * (rng.random(B.shape) < 0.1)
    tiny = B + 0.0
    tiny[::3] *= 1e-100
    ones = np.sign(B.real) + (1j * np.sign(B.imag) if cplx else 0)
    ident = np.eye(70, n) * 3 + 0 * B
    mats = [rows, cols, both, sparse, tiny, ones, ident]
    check(mats, run(mats, path), path)
    if path == "blocked":
        A = torch.from_numpy(np.stack([B, ones])).cuda()
        r = bsvd.gesvj(A, path="blocked", nb=16, flags=bsvd.FLAG_NO_MASKS)
        check([B, ones], [r.S.cpu().numpy(), r.U.cpu().numpy(), r.V.cpu().numpy(), r.info.cpu().numpy()], "no masks")


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("nb", [8, 16])
def test_on_chip_equals_slots_bitwise(nb, cplx):
    """The same tiles and the same order of sums on chip and in global slots, also
    for a single pair of blocks (all the CTA's threads in one group on chip)."""
    rng = np.random.default_rng(7)
    shapes = ((64, 50), (30, 48), (33, 40), (40, 25), (40, 13)) if cplx else ((64, 64), (90, 50), (33, 70), (40, 25), (40, 13))
    mats = [normal(rng, s, cplx) for s in shapes]
    a, b = run(mats, "fused", nb), run(mats, "slots", nb)
    for k in range(len(mats)):
        assert all(np.array_equal(a[i][k], b[i][k]) for i in range(3)), k


@pytest.mark.parametrize("cplx", [False, True])
def test_error_no_larger_than_on_the_fp64_pipe(cplx):
    """The product U S V^T of a full solve against 64-bit inputs: the digit
    products (nb = 16) stay within 1.5 times the error of the FP64 pipe's sums
    (nb = 32, the same path)."""
    rng = np.random.default_rng(8)
    for mats in ([rng.random((160, 160)) + (1j * rng.random((160, 160)) if cplx else 0) for _ in range(4)],
                 [normal(rng, (200, 96), cplx) for _ in range(4)]):
        A = torch.from_numpy(np.stack(mats)).cuda()
        err = []
        for nb in (16, 32):
            r = bsvd.gesvj(A, path="blocked", nb=nb)
            P = ((r.U * r.S[:, None, :]) @ r.V.mH).cpu().numpy()
            err.append(float(np.linalg.norm(P - np.stack(mats)) / np.linalg.norm(np.stack(mats))))
        assert err[0] <= 1.5 * err[1] + 4 * U, err
