"""The 3xTF32 kernel over C blocks of many passes and over few C blocks (passes of one 16 x 8 tile
instead of three): blocks above 70 columns, thin and long ones, passes whose last rows or columns
are one wide, C_in; against the oracle, and the same bits for a block whatever its passes.

Tolerance: a product's operands keep 2 x 11 bits (relative 2^-21 per product of elements) and
are summed in FP32 over at most 96 inner elements (96 2^-24), the products of a block in an
FP32 pair; 1e-5 relative Frobenius leaves a factor of two."""
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


@pytest.mark.parametrize("m,n,k,nb", [(512, 512, 96, 2), (100, 100, 33, 6), (73, 97, 8, 5), (1, 300, 17, 9),
                                      (300, 1, 17, 9), (129, 16, 96, 7), (24, 193, 9, 7), (5, 5, 5, 3),
                                      (48, 48, 40, 60), (23, 23, 23, 50)])
@pytest.mark.parametrize("ta,tb,cin", [("N", "N", True), ("T", "T", False)])
def test_many_passes_vs_oracle(m, n, k, nb, ta, tb, cin):
    import torch
    rng = np.random.default_rng(m * 31 + n)
    nk = 4
    rs, ks, cs = (np.full(c, v, np.int32) for c, v in ((nb, m), (nk, k), (nb, n)))
    mk = lambda a, b, p: make_matrix(rng, a, b, *bernoulli_pattern(rng, len(a), len(b), p))
    A = mk(ks, rs, 0.7) if ta == "T" else mk(rs, ks, 0.7)
    B = mk(cs, ks, 0.7) if tb == "T" else mk(ks, cs, 0.7)
    C = mk(rs, cs, 0.6) if cin else None
    alpha, beta = (-0.75, 1.25) if cin else (1.0, 0.0)
    ref = oracle.multiply(A, B, C, alpha, beta, 0.0, ta, tb)
    plan = bst.multiply(to_lib(A), to_lib(B), None if C is None else to_lib(C), alpha, beta, 0.0, ta, tb,
                        bst.BST_TF32X3)
    torch.cuda.synchronize()
    assert rel_fro(plan.result.data[:plan.result.info[3]].cpu().numpy(), ref["data"]) <= 1e-5


def test_a_block_has_the_same_bits_in_every_pass_width():
    import torch
    rng = np.random.default_rng(8)
    m, n, k, nk = 40, 31, 23, 5
    size = lambda v, c: np.full(c, v, np.int32)
    grid = lambda r, c: [x.ravel().astype(np.int32) for x in np.meshgrid(range(r), range(c), indexing="ij")]
    a, b = rng.standard_normal(nk * m * k), rng.standard_normal(nk * k * n)
    out = []
    for nb in (1, 60):  # one C block; 3600 equal ones, which fill the device
        A = bst.Matrix.from_host(size(m, nb), size(k, nk), *grid(nb, nk), np.tile(a, nb))
        B = bst.Matrix.from_host(size(k, nk), size(n, nb), *grid(nk, nb),
                                 np.concatenate([np.tile(x, nb) for x in np.split(b, nk)]))
        plan = bst.multiply(A, B, precision=bst.BST_TF32X3)
        torch.cuda.synchronize()
        out.append(plan.result.data[:plan.result.info[3]].reshape(-1, m * n).clone())
    assert torch.equal(out[1], out[0].expand(3600, -1))
