"""The 3xTF32 kernel at the edges of its passes (16 x 24 outputs of a C block or of its
transpose, 8-wide chunks of the inner size): sizes around 8, 16 and 24, inner sizes around
multiples of 8, C blocks of more than 32 products, blocks that only C_in has; against the
oracle.

Tolerance: a product's operands keep 2 x 11 bits (relative 2^-21 per product of elements) and
are summed in FP32 over at most 48 inner elements (48 2^-24), the products of a block in an
FP32 pair; 1e-5 relative Frobenius leaves a factor of three."""
import numpy as np
import pytest

import oracle
from gpu_util import rel_fro, require_gpu, to_lib
from paper_1910_13555_gb300 import bst
from paper_1910_13555_gb300.workloads import bernoulli_pattern, make_matrix

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


SIZES = [(1, 1, 1), (5, 5, 5), (8, 16, 8), (9, 17, 9), (16, 24, 16), (17, 25, 7), (24, 16, 13),
         (25, 17, 23), (23, 23, 23), (33, 50, 40), (50, 33, 48), (3, 70, 15)]


@pytest.mark.parametrize("m,n,k", SIZES)
@pytest.mark.parametrize("ta,tb,cin", [("N", "N", False), ("T", "N", True), ("N", "T", True),
                                       ("T", "T", False)])
def test_tf32_passes_vs_oracle(m, n, k, ta, tb, cin):
    import torch
    rng = np.random.default_rng(m * 10007 + n * 101 + k)
    nm, nk, nn = 9, 45, 8  # up to 45 products a block
    rs, ks, cs = (np.full(c, v, np.int32) for c, v in ((nm, m), (nk, k), (nn, n)))
    mk = lambda a, b, p: make_matrix(rng, a, b, *bernoulli_pattern(rng, len(a), len(b), p))
    A = mk(ks, rs, 0.9) if ta == "T" else mk(rs, ks, 0.9)
    B = mk(cs, ks, 0.9) if tb == "T" else mk(ks, cs, 0.9)
    if cin:  # empty the last rows of op(A): their C blocks come from C_in alone
        keep = (A.cols if ta == "T" else A.rows) < nm - 2
        A = make_matrix(rng, A.row_sizes, A.col_sizes, A.rows[keep], A.cols[keep])
    C = mk(rs, cs, 0.7) if cin else None
    alpha, beta = (-0.75, 1.25) if cin else (1.0, 0.0)
    ref = oracle.multiply(A, B, C, alpha, beta, 0.0, ta, tb)
    lA, lB, lC = to_lib(A), to_lib(B), None if C is None else to_lib(C)
    plan = bst.multiply(lA, lB, lC, alpha, beta, 0.0, ta, tb, bst.BST_TF32X3)
    got = plan.result.data[:plan.result.info[3]].clone()
    plan.result.data.fill_(float("nan"))
    plan.execute(alpha, beta, bst.BST_TF32X3)
    torch.cuda.synchronize()
    assert torch.equal(got, plan.result.data[:len(got)])
    assert rel_fro(got.cpu().numpy(), ref["data"]) <= 1e-5
