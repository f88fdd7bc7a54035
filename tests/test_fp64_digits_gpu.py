"""FP64 Gram blocks and updates as exact digit products on the tensor cores
(nb = 16; needs a GB300): on chip, multi-kernel, persistent in global slots.
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


def run(mats, path, **kw):
    T = [torch.from_numpy(np.ascontiguousarray(x.T)).cuda().t() for x in mats]
    if path == "slots":
        r = bsvd.gesvj_batched(T, path="persistent", nb=16, flags=bsvd.FLAG_NO_ONCHIP, **kw)
    else:
        r = bsvd.gesvj_batched(T, path=path, nb=16, **kw)
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


@pytest.mark.parametrize("path", ["fused", "blocked", "slots"])
def test_shapes(path):
    rng = np.random.default_rng(5)
    mats = [rng.standard_normal(s) for s in SHAPES]
    check(mats, run(mats, path), path)


@pytest.mark.parametrize("path", ["fused", "blocked", "slots"])
def test_exponent_ranges(path):
    """Rows and columns scaled over hundreds of binary orders, tiny and zero
    entries, equal magnitudes, and blocks in which J = I is applied (no masks)."""
    rng = np.random.default_rng(6)
    n = 48
    B = rng.standard_normal((70, n))
    rows = B * 2.0 ** -np.linspace(0, 300, 70).round()[:, None]
    cols = B * 2.0 ** -np.linspace(0, 60, n).round()
    both = rows * 2.0 ** -np.linspace(0, 60, n).round()
    sparse = B * (rng.random(B.shape) < 0.1)
    tiny = B + 0.0
    tiny[::3] *= 1e-100
    ones = np.sign(B)
    ident = np.eye(70, n) * 3
    mats = [rows, cols, both, sparse, tiny, ones, ident]
    check(mats, run(mats, path), path)
    if path == "blocked":
        A = torch.from_numpy(np.stack([B, ones])).cuda()
        r = bsvd.gesvj(A, path="blocked", nb=16, flags=bsvd.FLAG_NO_MASKS)
        check([B, ones], [r.S.cpu().numpy(), r.U.cpu().numpy(), r.V.cpu().numpy(), r.info.cpu().numpy()], "no masks")


def test_on_chip_equals_slots_bitwise():
    """The same tiles and the same order of sums on chip and in global slots, also
    for a single pair of blocks (all the CTA's threads in one group on chip)."""
    rng = np.random.default_rng(7)
    mats = [rng.standard_normal(s) for s in ((64, 64), (90, 50), (33, 70), (40, 25))]
    a, b = run(mats, "fused"), run(mats, "slots")
    for k in range(len(mats)):
        assert all(np.array_equal(a[i][k], b[i][k]) for i in range(3)), k


def test_error_no_larger_than_on_the_fp64_pipe():
    """The product U S V^T of a full solve against 64-bit inputs: the digit
    products (nb = 16) stay within 1.5 times the error of the FP64 pipe's sums
    (nb = 32, the same path)."""
    rng = np.random.default_rng(8)
    for mats in ([rng.random((160, 160)) for _ in range(4)], [rng.standard_normal((200, 96)) for _ in range(4)]):
        A = torch.from_numpy(np.stack(mats)).cuda()
        err = []
        for nb in (16, 32):
            r = bsvd.gesvj(A, path="blocked", nb=nb)
            P = ((r.U * r.S[:, None, :]) @ r.V.mT).cpu().numpy().astype(np.longdouble)
            err.append(float(np.linalg.norm((P - np.stack(mats)).astype(float)) / np.linalg.norm(np.stack(mats))))
        assert err[0] <= 1.5 * err[1] + 4 * U, err
