"""FP64 matrices of one block pair (needs a GB300): the preconditioned start only
with nb = 8 and from 24 rows a column on; below that line it made one 128 x 16 a
fifth slower.  Without it such a matrix takes the sweeps of inner_sweeps = 1, which
never starts preconditioned: the same bits."""
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


@pytest.mark.parametrize("dtype", [np.float64, np.complex128])
@pytest.mark.parametrize("m,n,nb,plain", [(128, 16, 8, True), (383, 16, 8, True), (100, 5, 8, True), (160, 20, 16, True),
                                          (256, 32, 16, True), (384, 16, 8, False), (120, 5, 8, False)])
def test_start_of_one_block_pair(m, n, nb, plain, dtype):
    rng = np.random.default_rng(m + n)
    cplx = np.issubdtype(dtype, np.complexfloating)
    A = (rng.standard_normal((4, m, n)) + (1j * rng.standard_normal((4, m, n)) if cplx else 0)).astype(dtype)
    if cplx and 16 * m * n > 100_000:
        pytest.skip("not on chip")
    T = torch.from_numpy(A).cuda()
    r, p = bsvd.gesvj(T, nb=nb, path="fused"), bsvd.gesvj(T, nb=nb, path="fused", inner_sweeps=1)
    torch.cuda.synchronize()
    assert torch.equal(r.U, p.U) == plain and torch.equal(r.V, p.V) == plain
    S, U, V = r.S.cpu().numpy(), r.U.cpu().numpy(), r.V.cpu().numpy()
    ref = oracle.gesvj(list(A))["S"]
    for k in range(4):
        assert int(r.info[k]) == 0
        assert checks.violations(checks.measures(A[k], S[k], U[k], V[k], ref[k]), checks.unit_roundoff(dtype)) == [], k
