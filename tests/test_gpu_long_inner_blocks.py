"""Inner block sizes around what a staged entry's strides hold (A's stored row length in 16 bits,
B's in 15): the staged kernel runs every plan whose stored rows fit, the direct-load kernel the
others, both against the oracle.

Tolerance: sums of at most 70 013 products, error below K 2^-53 relative to sum |a||b| (8e-12) and
about its square root in practice; 1e-12 relative Frobenius."""
import numpy as np
import pytest

import oracle
from gpu_util import rel_fro, require_gpu, to_lib
from helpers import random_matrix
from paper_1910_13555_gb300 import bst

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


# largest stored row length k that the strides hold
FITS = {("N", "N"): 65535, ("T", "N"): 1 << 30, ("N", "T"): 32767, ("T", "T"): 32767}


@pytest.mark.parametrize("big", [32767, 32768, 65535, 65536, 70001])
@pytest.mark.parametrize("ta,tb", FITS)
def test_route_and_result(ta, tb, big):
    import torch
    rng = np.random.default_rng(big)
    m, k, n = np.array([2, 3, 1], np.int32), np.array([big, 5, 7], np.int32), np.array([4, 2], np.int32)
    A = random_matrix(rng, k, m, 1.0) if ta == "T" else random_matrix(rng, m, k, 1.0)
    B = random_matrix(rng, n, k, 1.0) if tb == "T" else random_matrix(rng, k, n, 1.0)
    ref = oracle.multiply(A, B, None, 1.0, 0.0, 0.0, ta, tb)
    plan = bst.multiply(to_lib(A), to_lib(B), None, 1.0, 0.0, 0.0, ta, tb)
    torch.cuda.synchronize()
    assert plan.schedule_info()["staged"] == (big <= FITS[ta, tb])
    got = plan.result.data[:plan.result.info[3]].cpu().numpy()
    assert rel_fro(got, ref["data"]) <= 1e-12


@pytest.mark.parametrize("nP,nu", [(300, 130), (1100, 70), (9, 8000)])
def test_slabs_of_a_long_contracted_block(nP, nu):
    """T(P, mu, nu) contracted over (P, nu): inner blocks of P nu elements, read in place as slabs
    whose rows have nu."""
    import torch
    from paper_1910_13555_gb300.workloads import _tensor
    rng = np.random.default_rng(nP)
    one = np.zeros((1, 3), np.int64)
    T = _tensor(rng, [np.array([v], np.int32) for v in (nP, 5, nu)], one)
    U = _tensor(rng, [np.array([v], np.int32) for v in (nP, nu, 4)], one)
    lib = lambda t: bst.Tensor.from_host(t.block_sizes, t.index, t.data)
    keep = lib(T), lib(U)
    plan = bst.contract_plan(*keep, [0, 2], [0, 1], [1], [2], None, None, 0.0)
    plan.alloc_result()
    info = plan.schedule_info()
    assert info["staged"] and info["slab"]
    plan.execute(1.0, 0.0)
    torch.cuda.synchronize()
    ref = oracle.contract(T, U, [0, 2], [0, 1], [1], [2])
    assert rel_fro(plan.result.data[:plan.result.info[2]].cpu().numpy(), ref["data"]) <= 1e-12
