"""HITS and eigenvector centrality of small graphs, a launch a product: row lengths
at the edges of the kernel's cases against the FP64 oracle and the blocked
schedule, and vectors whose scale runs away between products."""
import numpy as np
import pytest

import oracle
import paper_1606_07550_gb300 as gpr
from test_pagerank_small import star_rows

pytestmark = pytest.mark.gpu


def vectors(torch, g, iters, spmv="auto"):
    h, a, x = (torch.empty(g.n, dtype=torch.float32, device="cuda") for _ in range(3))
    gpr.hits(g, h, a, iters=iters, spmv=spmv)
    gpr.eigen_centrality(g, x, iters=iters, spmv=spmv)
    return [v.cpu().numpy().astype(np.float64) for v in (h, a, x)]


@pytest.mark.parametrize("n,extra", [(1, 0), (33, 40), (1000, 5000), (16_400, 20_000), (70_001, 500_000)])
def test_row_lengths(n, extra):
    import torch
    src, dst = star_rows(n, extra, np.random.default_rng(n + 1))
    g = gpr.graph_build(src, dst, n)
    ref = oracle.build_csc(n, src, dst)
    for iters in (0, 1, 6):
        got = vectors(torch, g, iters)
        rh, ra = oracle.hits(ref, iters)
        rx = oracle.eigen_centrality(ref, iters)
        # FP32 products of non-negative terms: a relative error of at most a few
        # 2^-24 per product and in-edge block; 1e-5 as for the larger graphs
        for v, r in zip(got, (rh, ra, rx)):
            assert np.linalg.norm(v - r) <= 1e-5
        for v, b in zip(got, vectors(torch, g, iters, "blocked")):
            assert np.linalg.norm(v - b) <= 2e-5
        for v, again in zip(got, vectors(torch, g, iters)):
            assert (v == again).all()


def test_a_layered_graph_that_empties_beside_a_cycle():
    # five complete layers of 200 nodes: the vector grows 200-fold a product and
    # then leaves the layers at once, with 200^-5 of it on a cycle of 3 nodes
    import torch
    w, layers = 200, 5
    src, dst = [], []
    for k in range(layers - 1):
        a, b = np.meshgrid(np.arange(w) + k * w, np.arange(w) + (k + 1) * w)
        src.append(a.ravel())
        dst.append(b.ravel())
    n = w * layers + 3
    c = np.arange(3) + w * layers
    src, dst = np.concatenate(src + [c]), np.concatenate(dst + [np.roll(c, 1)])
    g = gpr.graph_build(src.astype(np.int32), dst.astype(np.int32), n)
    ref = oracle.build_csc(n, src.astype(np.int32), dst.astype(np.int32))
    for iters in (3, 4, 5, 8):
        x = torch.empty(n, dtype=torch.float32, device="cuda")
        gpr.eigen_centrality(g, x, iters=iters)
        assert np.linalg.norm(x.cpu().numpy() - oracle.eigen_centrality(ref, iters)) <= 1e-5
