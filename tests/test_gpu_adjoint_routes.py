"""Which route each gradient of a plan takes, for the plans of test_gpu_adjoint_staged.py (whose
results that file compares with the oracle) and for plans that stay on the direct kernels."""
import numpy as np
import pytest

from gpu_util import require_gpu, to_lib
from helpers import random_matrix, transpose_matrix
from paper_1910_13555_gb300 import bst
from test_gpu_adjoint_staged import CASES, _without

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _info(A, B, ta="N", tb="N"):
    import torch
    lA, lB = to_lib(A), to_lib(B)
    plan = bst.multiply(lA, lB, None, 1.0, 0.0, 0.0, ta, tb)
    assert not any(bst.bst_plan_adjoint_info(plan.handle).values())  # before the first adjoint
    g = torch.ones(max(plan.result.info[3], 1), dtype=torch.float64, device="cuda")
    bst.bst_plan_adjoint(plan.handle, g, torch.empty_like(lA.data), torch.empty_like(lB.data), None, 1.0, 0.0)
    torch.cuda.synchronize()
    return bst.bst_plan_adjoint_info(plan.handle)


# staged and tiled, dA then dB; None: either
ROUTES = {
    "whole": (True, False, True, False),
    "row_tiles": (True, True, True, True),
    "rectangles_a": (True, True, None, None),
    "rectangles_b": (None, None, True, True),
    "long_inner_a": (True, True, None, None),
    "long_inner_b": (None, None, True, True),
    "empty_groups": (True, False, True, False),
}


@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("ta,tb", [("N", "N"), ("T", "T")])
def test_staged_plans(name, ta, tb):
    sm, sk, sn, nb, occ = CASES[name]
    rng = np.random.default_rng(11)
    m, k, n = (rng.choice(np.array(s, np.int32), c).astype(np.int32) for s, c in zip((sm, sk, sn), nb))
    A, B = random_matrix(rng, m, k, occ[0]), random_matrix(rng, k, n, occ[1])
    if name == "empty_groups":
        A = _without(A, B, rng, k, n)[0]
    info = _info(transpose_matrix(A) if ta == "T" else A, transpose_matrix(B) if tb == "T" else B, ta, tb)
    for got, want in zip(info.values(), ROUTES[name], strict=True):
        assert want is None or got == want


@pytest.mark.parametrize("sizes,nb", [((1,), 1), ((5, 13), 8), ((5, 13, 23), 40), ((32,), 60)])
def test_direct_plans(sizes, nb):
    # too few flops, or blocks that fill their lanes
    rng = np.random.default_rng(2)
    s = rng.choice(np.array(sizes, np.int32), nb).astype(np.int32)
    occ = 1.0 if nb in (1, 60) else 0.4
    assert not any(_info(random_matrix(rng, s, s, occ), random_matrix(rng, s, s, occ)).values())
