"""Matrices of exact low rank through the preconditioned start (needs a GB300):
constant, checkerboard, block-constant and integer matrices.  Bounds as in
test_parity_gpu."""
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


def matrices(m, n):
    rng = np.random.default_rng(m + n)
    i, j = np.arange(m)[:, None], np.arange(n)[None]
    return [np.ones((m, n)), np.full((m, n), 0.3), (i + j) % 2 * 1.0, 1.0 * (i * 4 // m == j * 4 // n),
            i * 4 // m + j * 3 // n + 0.0, 1.0 * rng.integers(1, 9, (m, 1)) * rng.integers(1, 9, (1, n)),
            1.0 * rng.integers(-3, 4, (m, 3)) @ rng.integers(-3, 4, (3, n))]


@pytest.mark.parametrize("dtype", [np.float32, np.float64, np.complex64, np.complex128])
@pytest.mark.parametrize("m,n,nb", [(96, 96, 16), (64, 64, 16), (128, 64, 16), (150, 140, 16), (60, 40, 16), (60, 40, 8), (40, 90, 16)])
def test_low_rank(m, n, nb, dtype):
    if n == 140 and dtype in (np.float64, np.complex128):
        pytest.skip("the plain sweeps run into the sweep limit on the integer matrix of rank 3")
    mats = [x.astype(dtype) for x in matrices(m, n)]
    r = bsvd.gesvj_batched([torch.from_numpy(np.asfortranarray(x)).cuda() for x in mats], nb=nb, path="persistent")
    torch.cuda.synchronize()
    u = checks.unit_roundoff(dtype)
    wide = [x.astype(np.complex128 if np.iscomplexobj(x) else np.float64) for x in mats]
    ref = oracle.gesvj(wide)["S"]
    for k, A in enumerate(wide):
        assert int(r.info[k]) == 0, (k, int(r.info[k]))
        meas = checks.measures(A, r.S[k].cpu().numpy(), r.U[k].cpu().numpy(), r.V[k].cpu().numpy(), ref[k])
        # (the columns of W / sigma belong to noise and zeros: U, V of a wide matrix)
        gate = {"sigma_err", "resid", "orth_v" if m >= n else "orth_u"}
        assert not gate & set(checks.violations(meas, u)), (k, meas)
