"""Plan construction off its usual sizes, against the CPU oracle: enough size buckets and
products for the two-pass partition, inner block sizes around what the staged schedule takes
(2^15) and the class table holds (2^16), and plans built in turn on two streams (their uploads
share one staging buffer)."""
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


def _stacks_match(plan, ref):
    st = plan.stacks()
    return all((st[k] == ref[k]).all() for k in ("a_off", "b_off", "c_off", "bucket_ptr"))


def test_many_buckets_stacks_are_exact():
    rng = np.random.default_rng(3)
    # 40^3 buckets, about 200 000 products: one pass would need segments of 1024 items
    m, k, n = (rng.permutation(np.repeat(np.arange(1, 41, dtype=np.int32), 2))[:70] for _ in range(3))
    A, B = random_matrix(rng, m, k, 0.8), random_matrix(rng, k, n, 0.8)
    ref = oracle.multiply(A, B)
    plan = bst.multiply(to_lib(A), to_lib(B))
    assert plan.stats()["n_stack"] > 135000
    assert _stacks_match(plan, ref)
    got = plan.result.data[:plan.result.info[3]].cpu().numpy()
    assert rel_fro(got, ref["data"]) <= 1e-12


@pytest.mark.parametrize("big", [32767, 32768, 65536, 65537, 70001])
def test_block_sizes_around_the_class_table(big):
    rng = np.random.default_rng(4)
    m, k, n = np.array([2, 3, 1], np.int32), np.array([big, 5, 7], np.int32), np.array([4, 2], np.int32)
    A, B = random_matrix(rng, m, k, 1.0), random_matrix(rng, k, n, 1.0)
    ref = oracle.multiply(A, B)
    plan = bst.multiply(to_lib(A), to_lib(B))
    assert _stacks_match(plan, ref)
    got = plan.result.data[:plan.result.info[3]].cpu().numpy()
    assert rel_fro(got, ref["data"]) <= 1e-12


def test_plans_built_in_turn_on_two_streams():
    import torch
    rng = np.random.default_rng(5)
    sizes = [np.array(s, np.int32) for s in ((5,), (5, 13), (1, 2, 3, 40), (23,))]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    todo = []
    for q in range(12):
        s = rng.choice(sizes[q % 4], 20 + 30 * (q % 3)).astype(np.int32)
        A, B = random_matrix(rng, s, s, 0.2), random_matrix(rng, s, s, 0.2)
        todo.append((to_lib(A), to_lib(B), oracle.multiply(A, B)))
    torch.cuda.synchronize()
    plans = []
    for q, (A, B, _) in enumerate(todo):
        with torch.cuda.stream(streams[q % 2]):
            plans.append(bst.multiply(A, B))
    torch.cuda.synchronize()
    for plan, (_, _, ref) in zip(plans, todo):
        assert _stacks_match(plan, ref)
        got = plan.result.data[:plan.result.info[3]].cpu().numpy()
        assert rel_fro(got, ref["data"]) <= 1e-12
