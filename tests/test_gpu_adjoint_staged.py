"""The staged route of the adjoint (plans of at least 5e8 flops whose gradient blocks leave
lanes of the direct kernels idle: both sides or, "_a" and "_b", that one) against the CPU oracle's
adjoint: gradient blocks kept whole, cut into row tiles and into rectangular tiles, inner dimensions
cut into panels, every operand layout, blocks without products (zero gradient).

Tolerance: every gradient element is an FP64 sum of at most 1e5 products in some order,
error below K 2^-53 relative to sum |a||b|; 1e-12 relative Frobenius leaves ample room."""
import numpy as np
import pytest

import oracle
from gpu_util import rel_fro, require_gpu, to_lib
from helpers import random_matrix, transpose_matrix
from paper_1910_13555_gb300 import bst

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


CASES = {
    # (m sizes, k sizes, n sizes, block counts, occupancies)
    "whole": ((5, 13), (5, 13), (5, 13), (110, 110, 110), (0.55, 0.55)),
    "row_tiles": ((5, 13, 23), (5, 13, 23), (5, 13, 23), (90, 90, 90), (0.4, 0.4)),
    "rectangles_a": ((3, 5), (7, 110), (1, 17, 60), (90, 60, 70), (0.6, 0.6)),
    "rectangles_b": ((1, 17, 60), (7, 110), (3, 5), (70, 60, 90), (0.6, 0.6)),
    "long_inner_a": ((3, 5), (5, 13), (350, 9), (90, 60, 60), (0.5, 0.5)),
    "long_inner_b": ((350, 9), (5, 13), (3, 5), (60, 60, 90), (0.5, 0.5)),
    "empty_groups": ((5, 13), (5, 13), (5, 13), (130, 160, 130), (0.5, 0.5)),
}


@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("ta,tb", [("N", "N"), ("T", "N"), ("N", "T"), ("T", "T")])
def test_staged_adjoint_vs_oracle(name, ta, tb):
    import torch
    sm, sk, sn, nb, occ = CASES[name]
    rng = np.random.default_rng(11)
    m, k, n = (rng.choice(np.array(s, np.int32), c).astype(np.int32)
               for s, c in zip((sm, sk, sn), nb))
    A = random_matrix(rng, m, k, occ[0])
    B = random_matrix(rng, k, n, occ[1])
    if name == "empty_groups":  # the A blocks of these columns and B blocks of these rows
        A = _without(A, B, rng, k, n)[0]
    if ta == "T":
        A = transpose_matrix(A)
    if tb == "T":
        B = transpose_matrix(B)
    alpha = 1.0 if ta == tb else -0.75
    ref = oracle.multiply(A, B, None, alpha, 0.0, 0.0, ta, tb)
    G = rng.standard_normal(len(ref["data"]))
    rA, rB, _ = oracle.multiply_adjoint(A, B, None, alpha, 0.0, 0.0, G, ta, tb)
    lA, lB = to_lib(A), to_lib(B)
    plan = bst.multiply(lA, lB, None, alpha, 0.0, 0.0, ta, tb)
    assert plan.stats()["flops"] >= 5e8
    g = torch.as_tensor(G).cuda()
    got = []
    for _ in range(2):  # the first call builds the schedule
        dA, dB = torch.full_like(lA.data, np.nan), torch.full_like(lB.data, np.nan)
        bst.bst_plan_adjoint(plan.handle, g, dA, dB, None, alpha, 0.0)
        got.append((dA, dB))
    torch.cuda.synchronize()
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    assert rel_fro(got[0][0].cpu().numpy(), rA) <= 1e-12
    assert rel_fro(got[0][1].cpu().numpy(), rB) <= 1e-12


def _without(A, B, rng, k, n):
    """A with its first 40 block columns emptied, so that B's blocks there have no product."""
    from paper_1910_13555_gb300.workloads import make_matrix
    keep = A.cols >= 40
    return make_matrix(rng, A.row_sizes, k, A.rows[keep], A.cols[keep]), B
