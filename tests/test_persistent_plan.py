"""Where a persistent batch's matrices live (host-side plan, no GPU): FP64 matrices
whose W and V fit in shared memory only beside the digit products' smaller groups
run on chip while there is at most one matrix an SM, in global slots beyond."""
import pytest

import __graft_entry__  # noqa: F401
import paper_2601_17979_gb300 as bsvd


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()


@pytest.mark.parametrize("shape", [(64, 64), (61, 61)])
def test_shapes_in_between(shape):
    for count, where in ((1, 1), (100, 1), (2000, 0)):
        assert set(bsvd.persistent_plan("d", [shape] * count)[1].tolist()) == {where}, count


@pytest.mark.parametrize("dtype,shape", [("d", (56, 56)), ("d", (64, 40)), ("z", (46, 46)), ("s", (64, 64))])
def test_other_shapes_stay_on_chip(dtype, shape):
    for count in (1, 2000):
        assert set(bsvd.persistent_plan(dtype, [shape] * count)[1].tolist()) == {1}, count
