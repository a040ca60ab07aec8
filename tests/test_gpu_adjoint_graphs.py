"""Adjoint launches captured into CUDA graphs: more of them than a plan has work counters, replays
of two graphs of one plan that overlap, a replay with new values; the bits of an uncaptured call."""
import numpy as np
import pytest

from gpu_util import require_gpu, to_lib
from helpers import random_matrix
from paper_1910_13555_gb300 import bst

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def test_more_captured_adjoints_than_counters():
    import torch
    rng = np.random.default_rng(5)
    sz = lambda c: rng.choice(np.array((5, 13, 23), np.int32), c).astype(np.int32)
    m, k, n = sz(90), sz(90), sz(90)
    lA, lB = to_lib(random_matrix(rng, m, k, 0.4)), to_lib(random_matrix(rng, k, n, 0.4))
    plan = bst.multiply(lA, lB)
    assert plan.stats()["flops"] >= 5e8  # from here on the staged route
    g = torch.randn(plan.result.info[3], dtype=torch.float64, device="cuda")

    def adjoint(out):
        bst.bst_plan_adjoint(plan.handle, g, out[0], out[1], None, 1.0, 0.0)

    new = lambda: (torch.full_like(lA.data, np.nan), torch.full_like(lB.data, np.nan))
    want = new()
    adjoint(want)
    torch.cuda.synchronize()
    graphs = []
    for calls in (20, 20, 3):  # 86 launches: the third graph's have no counter of their own
        graph, side, outs = torch.cuda.CUDAGraph(), torch.cuda.Stream(), [new() for _ in range(calls)]
        with torch.cuda.graph(graph, stream=side):
            for out in outs:
                adjoint(out)
        graphs.append((graph, torch.cuda.Stream(), outs))
    for again in range(2):
        for _, _, outs in graphs:
            for out in outs:
                out[0].fill_(np.nan), out[1].fill_(np.nan)
        torch.cuda.synchronize()
        for graph, stream, _ in graphs:  # replays overlap
            with torch.cuda.stream(stream):
                graph.replay()
        torch.cuda.synchronize()
        for _, _, outs in graphs:
            for out in outs:
                assert torch.equal(out[0], want[0]) and torch.equal(out[1], want[1])
        g.mul_(2.0)  # the graphs read the current values
        adjoint(want)
        torch.cuda.synchronize()

