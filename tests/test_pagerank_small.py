"""PageRank of small graphs in one launch: rows at the edges of its cases (slices
of 32 rows, groups of 8 indices, long rows and their chunks), sizes on both
sides of the cluster's limit, against the FP64 oracle and the pull schedule's
kernels (which a warm start from the uniform vector takes)."""
import numpy as np
import pytest

import oracle
import paper_1606_07550_gb300 as gpr

from gpu_util import l1

pytestmark = pytest.mark.gpu


def tolerance(dt, iters, d=0.85):
    # BF16 rounds each contribution by at most 2^-9 of itself, so a step moves at
    # most d 2^-9 of the mass (on a graph of a few nodes nothing averages out),
    # and each later step shrinks that by d
    return 1e-5 + (d * 2.0 ** -9 * (1 - d ** iters) / (1 - d) if dt == gpr.BF16 else 0.0)


DEGREES = [0, 1, 7, 8, 9, 15, 16, 17, 63, 64, 65, 255, 256, 257, 511, 513, 4095, 16_385, 20_000]


def star_rows(n, extra, rng):
    """Rows of the in-degrees above, and `extra` random edges."""
    src, dst = [], []
    for i, deg in enumerate(d for d in DEGREES if d < n - 1):
        v = (5 + 7 * i) % n
        s = rng.choice(n - 1, deg, replace=False)
        src.append(s + (s >= v))
        dst.append(np.full(deg, v))
    src.append(rng.integers(0, n, extra))
    dst.append(rng.integers(0, n, extra))
    return np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32)


def run(torch, g, iters, dt, warm=False, stats=False):
    x = torch.full((g.n,), 1.0 / g.n, dtype=torch.float32, device="cuda")
    st = gpr.pagerank(g, x, iters=iters, dtype=dt, warm_start=warm, stats=stats)
    return x.cpu().numpy(), st


@pytest.mark.parametrize("n,extra", [(1, 0), (2, 1), (31, 0), (33, 40), (1000, 5000), (16_000, 1000), (16_400, 0),
                                     (25_000, 60_000), (70_001, 500_000)])
@pytest.mark.parametrize("dt", [gpr.FP32, gpr.BF16])
def test_sizes_and_row_lengths(n, extra, dt):
    import torch
    src, dst = star_rows(n, extra, np.random.default_rng(n))
    g = gpr.graph_build(torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda(), n)
    ref = oracle.build_csc(n, src, dst)
    for iters in (0, 1, 2, 40):
        x, st = run(torch, g, iters, dt, stats=True)
        xr = oracle.pagerank(ref, 0.85, iters)
        assert l1(x, xr) <= tolerance(dt, iters)
        assert abs(st.mass - x.astype(np.float64).sum()) <= 1e-6
        assert abs(st.dangling - x.astype(np.float64)[ref.outdeg == 0].sum()) <= 1e-6
        # the general kernels, from the same start
        y, sy = run(torch, g, iters, dt, warm=True, stats=True)
        assert np.abs(x.astype(np.float64) - y).sum() <= 2 * tolerance(dt, iters)
        assert abs(st.residual_l1 - sy.residual_l1) <= 2 * tolerance(dt, iters)
        # the same bits again, with and without stats
        assert (run(torch, g, iters, dt)[0] == x).all()


def test_other_damping_and_two_graphs_in_turn():
    import torch
    rng = np.random.default_rng(8)
    graphs = []
    for n, m in ((300, 2000), (40_000, 300_000)):
        src, dst = rng.integers(0, n, m).astype(np.int32), rng.integers(0, n, m).astype(np.int32)
        graphs.append((gpr.graph_build(src, dst, n), oracle.build_csc(n, src, dst)))
    for d in (0.5, 0.99):
        outs = []
        for g, _ in graphs * 2:  # nothing waits between the calls
            x = torch.empty(g.n, dtype=torch.float32, device="cuda")
            gpr.pagerank(g, x, damping=d, iters=30)
            outs.append(x)
        for (g, ref), x in zip(graphs * 2, outs):
            assert l1(x.cpu().numpy(), oracle.pagerank(ref, d, 30)) <= 1e-5


@pytest.mark.parametrize("n", [700_001, 1_300_003])
def test_sums_over_many_equal_rows(n):
    # All ranks but two are equal: a lane's two-float sum is exact to 2^-45 of
    # itself, the warp trees of equal numbers are exact, the two warps with other
    # ranks round by 5 * 2^-24 of their 20 * 32 / n of the mass, and 2^-60 is cut
    # off in each of 2 * 3,648 places: below 1e-9 together
    import torch
    g = gpr.graph_build(np.array([5], np.int32), np.array([9], np.int32), n)
    for iters in (0, 1, 3):
        x, st = run(torch, g, iters, gpr.FP32, stats=True)
        x = x.astype(np.float64)
        assert abs(st.mass - x.sum()) <= 1e-9 and abs(st.dangling - (x.sum() - x[5])) <= 1e-9


@pytest.mark.parametrize("n,m,one", [((3 << 19) + 100, 100, True), ((3 << 19) + 101, 100, False),
                                     (1 << 22, 3 << 20, True), ((1 << 22) + 1, 3 << 20, False)])
def test_lines_of_the_single_launch(n, m, one):
    # many rows for their edges: on both sides of the rule's lines, one launch a
    # call or the pull kernels, and the same ranks
    import torch
    gen = torch.Generator(device="cuda").manual_seed(n)
    dst = torch.randperm(n, dtype=torch.int32, device="cuda", generator=gen)[:m]  # m distinct edges
    g = gpr.graph_build((dst + 1) % n, dst, n)
    assert g.info().m == m
    x, _ = run(torch, g, 20, gpr.FP32)
    before = gpr.lib().gpr_kernel_launches()
    again, _ = run(torch, g, 20, gpr.FP32)
    assert (gpr.lib().gpr_kernel_launches() - before == 1) == one
    assert (again == x).all()
    y, _ = run(torch, g, 20, gpr.FP32, warm=True)
    assert l1(x, y) <= 2 * tolerance(gpr.FP32, 20)
    h, a = (torch.empty(n, device="cuda") for _ in range(2))
    gpr.hits(g, h, a, iters=2, spmv="pull")
    # an edge's head has one in-edge, its tail one out-edge: all hubs and authorities alike
    want = torch.zeros(n, device="cuda")
    want[dst.long()] = m ** -0.5
    assert float((a - want).norm()) <= 1e-5 and float((h - want.roll(1)).norm()) <= 1e-5


def test_tuner_times_the_single_launch():
    # the pull schedule of a small graph is timed as a call runs it: the same time
    # within a half (the pull kernels take more than twice as long here)
    import torch
    n, m = 180_000, 2_500_000
    gen = torch.Generator(device="cuda").manual_seed(4)
    src, dst = (torch.randint(0, n, (m,), dtype=torch.int32, device="cuda", generator=gen) for _ in range(2))
    g = gpr.graph_build(src, dst, n)
    x = torch.empty(n, dtype=torch.float32, device="cuda")
    r = gpr.pagerank_tune(g, trial_steps=100)
    best = min(gpr.pagerank(g, x, iters=100, spmv="pull", stats=True).t_iter_ms for _ in range(5))
    assert r.pull_ms_per_step * 100 <= 1.5 * best
    assert r.schedule == gpr.SPMV_PULL and r.ms_per_step == r.pull_ms_per_step
    before = gpr.lib().gpr_kernel_launches()
    gpr.pagerank(g, x, iters=100)
    assert gpr.lib().gpr_kernel_launches() - before == 1


def test_hub_of_equal_contributions():
    # every node points at node 0, which points back: one row of 23,074 equal
    # numbers, 64 chunks of 361 edges.  A chunk's sum rounds at most 3 times in a
    # lane's group, twice over its groups and 5 times over the warp, the chunks' 3 times
    # in an eight and 8 times over the eights, half an ulp of 2^-24 each, all the
    # same way: 0.85 * 21 * 2^-25; the start vector, the coefficients and the other
    # nodes (0.15 of the mass) round by 1.1e-7 together
    import torch
    n = 23_075
    o = np.arange(1, n, dtype=np.int32)
    z = np.zeros(n - 1, np.int32)
    src, dst = np.concatenate([o, z]), np.concatenate([z, o])
    g = gpr.graph_build(src, dst, n)
    x, _ = run(torch, g, 1, gpr.FP32)
    assert l1(x, oracle.pagerank(oracle.build_csc(n, src, dst), 0.85, 1)) <= 0.85 * 21 * 2.0 ** -25 + 1.1e-7
