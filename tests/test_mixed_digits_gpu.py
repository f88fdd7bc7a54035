"""The mixed path's restoration of V and A_hat in real FP64 as tiled digit
products (needs a GB300): edges of the 64 x 32 tiles and 32-term chunks, both
ends of FP64's range, entries that are not finite.  Bounds as in test_mixed_gpu."""
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


def mixed(mats):
    T = [torch.from_numpy(np.ascontiguousarray(x.T)).cuda().t() for x in mats]
    r = bsvd.gesvj_batched(T, prec="mixed", nb=16)
    torch.cuda.synchronize()
    return r


# one tile less a row, exact, one more; one chunk and one more; the last size
# with the preconditioning step and the first without; wide (A' = A^T)
SHAPES = [(1, 1), (2, 2), (31, 31), (33, 32), (63, 33), (64, 64), (65, 65), (97, 96), (128, 127), (129, 128), (161, 129),
          (40, 130), (129, 200), (300, 5)]


@pytest.mark.parametrize("exponent", [0, -1000, 1010])
def test_shapes_and_scales(exponent):
    rng = np.random.default_rng(11)
    mats = [rng.standard_normal(s) for s in SHAPES]
    r = mixed([np.ldexp(x, exponent) for x in mats])
    ref = oracle.gesvj(mats)["S"]
    for i, A in enumerate(mats):
        assert int(r.info[i]) == 0, A.shape
        meas = checks.measures(A, np.ldexp(r.S[i].cpu().numpy(), -exponent), r.U[i].cpu().numpy(), r.V[i].cpu().numpy(),
                               ref[i])
        assert checks.violations(meas, checks.U64) == [], (A.shape, meas)


def test_not_finite():
    rng = np.random.default_rng(12)
    mats = [rng.standard_normal((70, 66)) for _ in range(3)]
    mats[1][69, 0] = np.nan
    mats[2][3, 65] = np.inf
    r = mixed(mats)
    assert [int(x) == 0 for x in r.info] == [True, False, False]
    assert all(bool(torch.isnan(r.S[i]).all()) for i in (1, 2))
