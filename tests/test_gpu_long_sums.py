"""Rounding of long inner sums in the staged native-FP64 kernel, and a plan's bits alone and in a
batch.

Where a whole-tile split would pay, no tile may sum its outputs in one chain over the whole inner
dimension, whichever split it takes.  Tolerance: all terms are positive, so a chain's rounding
errors grow with its partial sums; two chains of half the length round as 1 / sqrt(2) = 0.71 of
one, more chains less.  One chain is formed here in float64 from the same values."""
import numpy as np
import pytest

from gpu_util import require_gpu
from paper_1910_13555_gb300 import bst

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _full(m, n, k, nb, kb, seed):
    """Dense pattern: nb x nb C blocks of m x n, each a sum of kb products of inner size k."""
    rng = np.random.default_rng(seed)
    grid = lambda r, c: [x.ravel().astype(np.int32) for x in np.meshgrid(range(r), range(c), indexing="ij")]
    a, b = rng.random((nb, kb, m, k)), rng.random((kb, nb, k, n))
    size = lambda v, c: np.full(c, v, np.int32)
    A = bst.Matrix.from_host(size(m, nb), size(k, kb), *grid(nb, kb), a.ravel())
    B = bst.Matrix.from_host(size(k, kb), size(n, nb), *grid(kb, nb), b.ravel())
    return A, B, a, b


@pytest.mark.parametrize("m,n,k,kb", [(10, 10, 35, 60), (5, 13, 35, 60), (13, 5, 35, 60),
                                      (12, 12, 35, 60), (13, 13, 35, 60), (9, 9, 35, 60),
                                      (7, 7, 35, 60), (5, 23, 35, 60), (10, 10, 13, 60),
                                      (5, 13, 13, 60), (5, 13, 35, 2)])
def test_no_single_chain(m, n, k, kb):
    import torch
    A, B, a, b = _full(m, n, k, 8, kb, seed=m * n + k)
    plan = bst.multiply(A, B)
    torch.cuda.synchronize()
    got = plan.result.data[:plan.result.info[3]].cpu().numpy().reshape(8, 8, m, n)
    err = chain = 0.0
    for i, j in ((0, 0), (2, 5), (4, 3), (7, 6)):
        x = a[i].transpose(1, 0, 2).reshape(m, kb * k)
        y = b[:, j].reshape(kb * k, n)
        exact = np.zeros((m, n), np.longdouble)
        one = np.zeros((m, n))
        for l in range(kb * k):
            exact += x[:, l:l + 1].astype(np.longdouble) * y[l:l + 1].astype(np.longdouble)
            one += x[:, l:l + 1] * y[l:l + 1]
        err += float(((got[i, j] - exact) ** 2).sum())
        chain += float(((one - exact) ** 2).sum())
    assert err ** 0.5 <= 0.75 * chain ** 0.5


def test_batch_has_the_bits_of_its_plans():
    import torch
    # tail splits only; whole-tile splits; rows that take the wide shape; panels by themselves
    shapes = [(23, 23, 35, 20), (5, 5, 13, 60), (3, 400, 7, 20), (13, 13, 35, 20), (13, 13, 13, 20)]
    mats = [_full(m, n, k, 6, kb, seed=i)[:2] for i, (m, n, k, kb) in enumerate(shapes)]
    plans = [bst.multiply_plan(A, B) for A, B in mats]
    outs = [p.alloc_result() for p in plans]
    for p in plans:
        p.execute(1.0, 0.0)
    torch.cuda.synchronize()
    alone = [C.data.clone() for C in outs]
    for C in outs:
        C.data.fill_(float("nan"))
    batch = bst.bst_batch_create(bst.context(), [p.handle for p in plans])
    bst.bst_batch_execute(batch, [1.0] * len(plans), [0.0] * len(plans))
    torch.cuda.synchronize()
    for C, want in zip(outs, alone):
        n = C.info[3]
        assert torch.equal(C.data[:n], want[:n])
    bst.bst_batch_destroy(batch)
