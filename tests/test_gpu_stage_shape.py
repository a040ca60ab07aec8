"""Which shape of the staged native-FP64 kernel a plan takes, seen in the inner splits that only the
wide one has room for (544 partial sums a tile against 320), and its results against the oracle.

Tolerance: every output is an FP64 sum of at most 2100 products in some order, error below
K 2^-53 relative to sum |a||b|; 1e-12 relative Frobenius leaves ample room."""
import numpy as np
import pytest

import oracle
from gpu_util import rel_fro, require_gpu, run_multiply
from paper_1910_13555_gb300.workloads import Problem, make_matrix

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _dense(rng, m, n, k, nb, kb):
    size = lambda v, c: np.full(c, v, np.int32)
    grid = lambda r, c: [x.ravel().astype(np.int32) for x in np.meshgrid(range(r), range(c), indexing="ij")]
    return Problem(make_matrix(rng, size(m, nb), size(k, kb), *grid(nb, kb)),
                   make_matrix(rng, size(k, kb), size(n, nb), *grid(kb, nb)), None)


# (m, n, k, products per block): split of every tile in the wide shape
@pytest.mark.parametrize("m,n,k,kb,split", [(9, 9, 35, 60, 5), (7, 7, 35, 60, 7), (5, 23, 35, 60, 3),
                                            (23, 5, 35, 60, 3), (13, 13, 35, 60, 3)])
def test_long_sums_of_small_blocks_take_the_wide_shape(m, n, k, kb, split):
    p = _dense(np.random.default_rng(m + n), m, n, k, 9, kb)
    out = run_multiply(p, stacks=False)
    assert out["plan"].split_histogram()[split] == 81
    ref = oracle.multiply(p.A, p.B, None, 1.0, 0.0, 0.0)
    assert rel_fro(out["data"], ref["data"]) <= 1e-12


# equal counts in both shapes, or a tail split that the narrow shape runs with a fourth CTA
@pytest.mark.parametrize("m,n,k,kb,split", [(5, 5, 35, 60, 5), (5, 13, 35, 60, 16), (9, 9, 13, 60, 1),
                                            (5, 13, 35, 2, 4)])
def test_others_stay_narrow(m, n, k, kb, split):
    p = _dense(np.random.default_rng(m + n), m, n, k, 9, kb)
    out = run_multiply(p, stacks=False)
    assert out["plan"].split_histogram()[split] == 81
    ref = oracle.multiply(p.A, p.B, None, 1.0, 0.0, 0.0)
    assert rel_fro(out["data"], ref["data"]) <= 1e-12


# rows of one tile each, whose slots hold panels of four elements: no split, no sum per panel (which
# the wide instance alone would add: "split" tells)
@pytest.mark.parametrize("m,n,k,kb", [(9, 200, 60, 6), (3, 200, 40, 6), (2, 199, 40, 6)])
def test_narrow_panels_of_row_tiles_keep_one_chain(m, n, k, kb):
    p = _dense(np.random.default_rng(n), m, n, k, 3, kb)
    out = run_multiply(p, stacks=False)
    assert not out["plan"].schedule_info()["split"]
    ref = oracle.multiply(p.A, p.B, None, 1.0, 0.0, 0.0)
    assert rel_fro(out["data"], ref["data"]) <= 1e-12


@pytest.mark.parametrize("k,products", [(200, 4), (60, 30), (49, 99)])
def test_fewer_products_than_blocks(k, products):
    """C blocks that only C_in has outnumber the products, whose inner sizes make long sums all the
    same on average."""
    rng = np.random.default_rng(k)
    size = lambda v, c: np.full(c, v, np.int32)
    grid = [x.ravel().astype(np.int32) for x in np.meshgrid(range(10), range(10), indexing="ij")]
    at = np.sort(rng.choice(100, products, replace=False)).astype(np.int32)
    A = make_matrix(rng, size(5, 10), size(k, 100), at // 10, at)  # one product each
    B = make_matrix(rng, size(k, 100), size(13, 10), np.arange(100, dtype=np.int32),
                    np.arange(100, dtype=np.int32) % 10)
    C = make_matrix(rng, size(5, 10), size(13, 10), *grid)
    out = run_multiply(Problem(A, B, C, alpha=1.0, beta=-2.0), stacks=False)
    ref = oracle.multiply(A, B, C, 1.0, -2.0, 0.0)
    assert out["stats"]["n_stack"] == products and len(out["rows"]) == 100
    assert rel_fro(out["data"], ref["data"]) <= 1e-12


def test_slab_reading_that_a_block_rules_out_keeps_the_narrow_shape():
    import torch
    from paper_1910_13555_gb300 import bst
    from paper_1910_13555_gb300.workloads import _tensor
    rng = np.random.default_rng(3)
    P, nu = np.full(6, 3, np.int32), np.full(5, 7, np.int32)
    mu = np.array([20, 24, 20, 24], np.int32)  # C blocks of 400 to 576 elements
    every = lambda *n: np.stack([x.ravel() for x in np.meshgrid(*map(range, n), indexing="ij")], 1)
    T, U = _tensor(rng, [P, mu, nu], every(6, 4, 5)), _tensor(rng, [P, nu, mu], every(6, 5, 4))
    lib = lambda t: bst.Tensor.from_host(t.block_sizes, t.index, t.data)
    keep = lib(T), lib(U)
    plan = bst.contract_plan(*keep, [0, 2], [0, 1], [1], [2], None, None, 0.0)
    plan.alloc_result()
    assert not plan.schedule_info()["slab"]
    assert plan.split_histogram().sum() == 2 * 16  # tiles of at most 320 elements
    plan.execute(1.0, 0.0)
    torch.cuda.synchronize()
    ref = oracle.contract(T, U, [0, 2], [0, 1], [1], [2])
    assert rel_fro(plan.result.data[:plan.result.info[2]].cpu().numpy(), ref["data"]) <= 1e-12


# AO sizes; the inner splits of the shape that their plans take
@pytest.mark.parametrize("sizes,splits", [((9,), {3}), ((7, 12), {2, 3, 7}), ((5, 13), {3, 5, 16}),
                                          ((17,), {16})])
def test_slab_reading_of_small_blocks(sizes, splits):
    import torch
    from paper_1910_13555_gb300 import bst
    from paper_1910_13555_gb300.workloads import _tensor
    rng = np.random.default_rng(4)
    P, ao = np.full(12, 30, np.int32), np.resize(np.array(sizes, np.int32), 8)
    every = np.stack([x.ravel() for x in np.meshgrid(range(12), range(8), range(8), indexing="ij")], 1)
    T, U = _tensor(rng, [P, ao, ao], every), _tensor(rng, [P, ao, ao], every)
    lib = lambda t: bst.Tensor.from_host(t.block_sizes, t.index, t.data)
    keep = lib(T), lib(U)
    plan = bst.contract_plan(*keep, [0, 2], [0, 1], [1], [2], None, None, 0.0)
    plan.alloc_result()
    assert plan.schedule_info()["slab"]
    assert set(np.nonzero(plan.split_histogram())[0]) == splits
    plan.execute(1.0, 0.0)
    torch.cuda.synchronize()
    ref = oracle.contract(T, U, [0, 2], [0, 1], [1], [2])
    assert rel_fro(plan.result.data[:plan.result.info[2]].cpu().numpy(), ref["data"]) <= 1e-12


@pytest.mark.parametrize("m,n,k,kb,warps", [(23, 23, 23, 60, 16), (9, 9, 35, 60, 12), (5, 13, 13, 60, 16)])
def test_automatic_k_split_counts_the_shape_s_warps(m, n, k, kb, warps):
    import torch
    p = _dense(np.random.default_rng(7), m, n, k, 40, kb)
    out = run_multiply(p, stacks=False, split_k=0)
    tiles = int(out["plan"].split_histogram().sum())
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    want = -(-sms * warps * 8 // tiles)
    assert out["stats"]["split_k"] == max(1, min(want, 1600 * kb // tiles, 16))
    ref = oracle.multiply(p.A, p.B, None, 1.0, 0.0, 0.0)
    assert rel_fro(out["data"], ref["data"]) <= 1e-12
