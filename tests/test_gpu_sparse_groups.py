"""Grouping of products by the blocks of an operand of which few take part (the adjoint groups by
stored block): operands of more than 2^24 blocks, long runs of blocks without products before,
between and after the others.

Tolerance: single products of 1 x 1 blocks, exact up to one rounding; 1e-15 relative."""
import numpy as np
import pytest

from gpu_util import require_gpu
from paper_1910_13555_gb300 import bst

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


# (rows, columns of A; the block rows of B that exist)
@pytest.mark.parametrize("nr,nc,used", [(4200, 4200, (0,)), (4200, 4200, (4199,)), (4200, 4200, (17, 2100)),
                                        (1500, 1400, (3,)), (9000, 1000, (0, 500, 999))])
def test_adjoint_with_few_products(nr, nc, used):
    import torch
    ones = lambda c: np.ones(c, np.int32)
    rows = np.repeat(np.arange(nr, dtype=np.int32), nc)
    cols = np.tile(np.arange(nc, dtype=np.int32), nr)
    rng = np.random.default_rng(nr + len(used))
    a, b = rng.standard_normal(nr * nc), rng.standard_normal(len(used))
    used = np.array(used, np.int32)
    A = bst.Matrix.from_host(ones(nr), ones(nc), rows, cols, a)
    B = bst.Matrix.from_host(ones(nc), ones(1), used, np.zeros(len(used), np.int32), b)
    plan = bst.multiply(A, B)
    assert plan.stats()["n_stack"] == nr * len(used)
    g = rng.standard_normal(nr)
    dA, dB = torch.full_like(A.data, np.nan), torch.full_like(B.data, np.nan)
    bst.bst_plan_adjoint(plan.handle, torch.as_tensor(g).cuda(), dA, dB, None, 1.0, 0.0)
    torch.cuda.synchronize()
    want = np.zeros((nr, nc))
    want[:, used] = g[:, None] * b[None, :]
    got = dA.cpu().numpy().reshape(nr, nc)
    assert np.abs(got - want).max() <= 1e-15 * np.abs(want).max()
    wb = a.reshape(nr, nc)[:, used].T @ g
    assert np.abs(dB.cpu().numpy()[:len(used)] - wb).max() <= 1e-11 * np.abs(wb).max()
