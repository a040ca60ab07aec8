"""The staged native-FP64 kernel at the edges of its tiles: outputs m n around multiples of
32 (the last partial round of lanes splits the inner dimension over lane groups), around
the 320-element tile (row tiles), operands around the 896-double slot (equal panels), a
C_in block read through the prefetch, transposed operands; against the oracle.

Tolerance: every output is an FP64 sum of at most a few thousand products in some order,
error below K 2^-53 relative to sum |a||b|; 1e-12 relative Frobenius leaves ample room."""
import numpy as np
import pytest

import oracle
from gpu_util import rel_fro, require_gpu, run_multiply
from paper_1910_13555_gb300.workloads import Problem, bernoulli_pattern, make_matrix

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _problem(m, n, k, ta, tb, cin, seed):
    rng = np.random.default_rng(seed)
    nb = 12
    rs, ks, cs = (np.full(nb, v, np.int32) for v in (m, k, n))
    mk = lambda a, b: make_matrix(rng, a, b, *bernoulli_pattern(rng, nb, nb, 0.35))
    A = mk(ks, rs) if ta else mk(rs, ks)
    B = mk(cs, ks) if tb else mk(ks, cs)
    C = mk(rs, cs) if cin else None
    return Problem(A, B, C, alpha=-0.75 if cin else 1.0, beta=1.25 if cin else 0.0,
                   transa="T" if ta else "N", transb="T" if tb else "N")


# m n mod 32: 1, 31, 0, 16, 17, 25, 9, 1 (one output), 1 row of 32, then tiles of 320, 321,
# 2 x 320 and one row more; slots of 896 and 897 doubles, panels of a long inner block;
# C rows of 321 to 544 elements (the wide shape)
SIZES = [(5, 13, 13), (9, 7, 5), (8, 8, 3), (4, 12, 23), (7, 7, 40), (5, 5, 1), (13, 13, 13),
         (1, 1, 29), (1, 32, 7), (3, 11, 2), (16, 20, 24), (3, 107, 8), (32, 20, 11),
         (33, 20, 11), (23, 23, 23), (32, 32, 14), (23, 23, 20), (13, 13, 35), (1, 320, 2),
         (2, 319, 5), (40, 40, 33), (2, 321, 5), (3, 400, 7), (1, 544, 3)]


@pytest.mark.parametrize("ta,tb,cin", [(False, False, False), (True, False, True),
                                       (False, True, True), (True, True, False)])
@pytest.mark.parametrize("m,n,k", SIZES)
def test_tile_edges(m, n, k, ta, tb, cin):
    p = _problem(m, n, k, ta, tb, cin, seed=m * 1000 + n * 10 + k)
    out = run_multiply(p, stacks=False)
    ref = oracle.multiply(p.A, p.B, p.C_in, p.alpha, p.beta, p.eps, p.transa, p.transb)
    assert (out["rows"] == ref["rows"]).all() and (out["cols"] == ref["cols"]).all()
    assert out["plan"].schedule_info()["staged"]
    assert rel_fro(out["data"], ref["data"]) <= 1e-12


def test_batch_of_both_shapes():
    import torch

    from gpu_util import to_lib
    from paper_1910_13555_gb300 import bst
    probs = [_problem(13, 23, 13, False, False, False, 1), _problem(3, 400, 7, False, False, False, 2),
             _problem(5, 13, 5, True, False, False, 3)]
    mats = [(to_lib(p.A), to_lib(p.B)) for p in probs]
    plans = [bst.multiply_plan(A, B, None, p.eps, p.transa, p.transb)
             for p, (A, B) in zip(probs, mats)]
    outs = [q.alloc_result() for q in plans]
    batch = bst.bst_batch_create(bst.context(), [q.handle for q in plans])
    bst.bst_batch_execute(batch, [1.0] * 3, [0.0] * 3)
    torch.cuda.synchronize()
    for p, C in zip(probs, outs):
        ref = oracle.multiply(p.A, p.B, None, 1.0, 0.0, p.eps, p.transa, p.transb)
        assert rel_fro(C.data[:C.info[3]].cpu().numpy(), ref["data"]) <= 1e-12
    bst.bst_batch_destroy(batch)
