"""A first 3xTF32 execute that is captured into a CUDA graph, in a context with its own allocator: the
replay must not touch memory that the library handed back while it was captured."""
import numpy as np
import pytest

import oracle
from gpu_util import rel_fro, require_gpu
from paper_1910_13555_gb300 import bst
from paper_1910_13555_gb300.workloads import bernoulli_pattern, make_matrix

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


class _Bump:
    """Every allocation has memory of its own; what is freed is remembered."""

    def __init__(self, nbytes):
        import torch
        self.buf = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")
        self.used = 0
        self.live, self.freed = {}, []

    def alloc(self, nbytes, user, stream):
        at = self.used
        self.used = at + (int(nbytes) + 255 & ~255)
        if self.used > self.buf.numel():
            return None
        self.live[self.buf.data_ptr() + at] = (at, int(nbytes))
        return self.buf.data_ptr() + at

    def free(self, ptr, user, stream):
        self.freed.append(self.live.pop(ptr))


def test_replay_leaves_freed_memory_alone():
    import torch
    rng = np.random.default_rng(3)
    s = np.full(9, 40, np.int32)  # several passes a block
    A, B = (make_matrix(rng, s, s, *bernoulli_pattern(rng, 9, 9, 0.6)) for _ in range(2))
    mem = _Bump(1 << 28)
    ctx = bst.bst_context_create(0, mem.alloc, mem.free)
    data = [torch.as_tensor(m.data).cuda() for m in (A, B)]
    mats = [bst.bst_matrix_create(ctx, m.row_sizes, m.col_sizes, m.rows, m.cols, d) for m, d in zip((A, B), data)]
    plan = bst.bst_multiply_plan(ctx, "N", "N", *mats, None, 0.0)
    C = bst.bst_plan_result(plan)
    out = torch.full((bst.bst_matrix_info(C)[3],), np.nan, dtype=torch.float64, device="cuda")
    bst.bst_matrix_bind_data(C, out)
    bst.bst_multiply_execute(plan, 1.0, 0.0, bst.BST_FP64_EMU_BF16, 1)  # what both share is built
    torch.cuda.synchronize()
    mem.freed.clear()
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=side):
        bst.bst_multiply_execute(plan, 1.0, 0.0, bst.BST_TF32X3, 1)
    for at, n in mem.freed:
        mem.buf[at:at + n] = 0xA5
    out.fill_(np.nan)
    graph.replay()
    torch.cuda.synchronize()
    for at, n in mem.freed:
        assert bool((mem.buf[at:at + n] == 0xA5).all())
    ref = oracle.multiply(A, B, None, 1.0, 0.0, 0.0)
    assert rel_fro(out.cpu().numpy(), ref["data"]) <= 1e-5
    del graph
    bst.bst_plan_destroy(plan)
    for m in mats:
        bst.bst_matrix_destroy(m)
    bst.bst_context_destroy(ctx)
