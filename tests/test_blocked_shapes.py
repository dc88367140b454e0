"""Blocked layouts of several shapes alive at once: a graph's steps run whatever
shapes were built after its own, and the ranks are those of the pull schedule."""
import os

import pytest

import gen
import paper_1606_07550_gb300 as gpr
from gpu_util import l1

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first, second", [("15,14", "15,12"), ("15,12", "15,14"), ("14,14", "12,10"), ("12,10", "15,13")])
def test_shapes_in_turn(first, second):
    n, m = 40_000, 400_000
    graphs = []
    for seed in (3, 4):
        src, dst = gen.rmat_coo(n, m, seed=seed)
        g = gpr.graph_build(torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda(), n)
        graphs.append(g)

    def ranks(g, iters, spmv):
        x = torch.empty(n, dtype=torch.float32, device="cuda")
        gpr.pagerank(g, x, iters=iters, spmv=spmv)
        return x.cpu().numpy()

    old = os.environ.get("GPR_BLOCK_BITS")
    try:
        for g, shape in zip(graphs, (first, second)):
            os.environ["GPR_BLOCK_BITS"] = shape
            ranks(g, 3, "blocked")
        os.environ["GPR_BLOCK_BITS"] = first
        for iters in (5, 8):  # new step counts: the steps are captured again
            x = ranks(graphs[0], iters, "blocked")
            # the bound that each schedule meets against the oracle
            assert l1(x, ranks(graphs[0], iters, "pull")) <= 1e-5
    finally:
        os.environ.pop("GPR_BLOCK_BITS", None)
        if old is not None:
            os.environ["GPR_BLOCK_BITS"] = old
    for g in graphs:
        g.free()
