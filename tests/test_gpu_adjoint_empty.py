"""Adjoint of products whose operands have no blocks, or no products: gradients of zero, or none."""
import numpy as np
import pytest

from gpu_util import require_gpu, to_lib
from paper_1910_13555_gb300 import bst
from paper_1910_13555_gb300.workloads import make_matrix

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("a,b", [(False, True), (True, False), (False, False), (True, True)])
def test_empty_operands(a, b):
    import torch
    rng = np.random.default_rng(1)
    s = np.array([3, 5, 2], np.int32)
    at = np.array([0, 1], np.int32)
    none = np.zeros(0, np.int32)
    A = make_matrix(rng, s, s, *((at, at) if a else (none, none)))  # rows 0, 1 meet no block of B
    B = make_matrix(rng, s, s, *((at[:1] + 2, at[:1]) if b else (none, none)))
    C = make_matrix(rng, s, s, at, at)
    lA, lB, lC = to_lib(A), to_lib(B), to_lib(C)
    plan = bst.multiply(lA, lB, lC, 1.0, 1.0)
    assert plan.stats()["n_stack"] == 0
    g = torch.ones(plan.result.info[3], dtype=torch.float64, device="cuda")
    dA, dB, dC = (torch.full_like(x.data, np.nan) for x in (lA, lB, lC))
    bst.bst_plan_adjoint(plan.handle, g, dA, dB, dC, 1.0, 2.0)
    torch.cuda.synchronize()
    for x, m in ((dA, A), (dB, B)):
        assert bool((x[:len(m.data)] == 0).all())
    assert bool((dC[:len(C.data)] == 2).all())
