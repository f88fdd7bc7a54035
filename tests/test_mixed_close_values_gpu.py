"""The mixed path on spectra of many nearly equal singular values (needs a
GB300): the first-order step of the restoration then has a large norm though
each of its entries is small.  Bounds as in test_mixed_gpu."""
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


def matrices(m, n):
    rng = np.random.default_rng(1000 * m + n)
    k = min(m, n)
    mats = [synth.with_sigma(rng, m, n, 1 + g * np.arange(k)) for g in (1e-7, 3e-7, 1e-6, 3e-6, 1e-5, 1e-4)]
    Q = synth.with_sigma(rng, m, n, np.ones(k))
    mats += [Q + eps * rng.standard_normal((m, n)) for eps in (1e-7, 1e-6, 1e-5, 1e-4)]
    mats += [synth.with_sigma(rng, m, n, synth.sigma_family(f, k, 1e4)) for f in ("cluster0", "cluster1")]
    return mats


@pytest.mark.parametrize("m,n", [(40, 33), (60, 40), (64, 64), (45, 97), (96, 96), (126, 126), (200, 127)])
@pytest.mark.parametrize("form", ["strided", "pointers"])
def test_close_values(form, m, n):
    mats = matrices(m, n)
    if form == "strided":
        r = bsvd.gesvj(torch.from_numpy(np.stack(mats)).cuda(), prec="mixed")
    else:
        r = bsvd.gesvj_batched([torch.from_numpy(np.asfortranarray(x)).cuda() for x in mats], prec="mixed")
    torch.cuda.synchronize()
    ref = oracle.gesvj(mats, tol=30 * checks.U64)["S"]
    for i, A in enumerate(mats):
        assert int(r.info[i]) == 0, i
        meas = checks.measures(A, r.S[i].cpu().numpy(), r.U[i].cpu().numpy(), r.V[i].cpu().numpy(), ref[i])
        assert checks.violations(meas, checks.U64) == [], (i, meas)
