"""The step-by-step schedule of batched personalised PageRank: rows at the edges of
its cases (short rows, blocks of 64 edges, long rows cut into chunks), every
width, each against the FP64 oracle and the cluster schedule, and the same bits
at every width."""
import os

import numpy as np
import pytest

import oracle
import paper_1606_07550_gb300 as gpr

from gpu_util import l1

DEGREES = [0, 1, 2, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 96, 127, 128, 129, 191, 192, 193, 255, 256, 257, 1023,
           1025, 4097, 32_767, 32_768, 32_769]
N = 33_000


def test_chunks_of_a_long_row_fit_the_list():
    # the chunk list holds edges / 64 entries: every long row must need at most
    # a 64th of its edges, and few enough chunks for one warp to add
    def chunk_edges(deg):
        c = 128
        while deg // c >= 2 * c:
            c *= 2
        return c
    for deg in list(range(129, 5000)) + [2 ** k + d for k in range(12, 31) for d in (-1, 0, 1)]:
        c = chunk_edges(deg)
        cnt = -(-deg // c)
        assert cnt <= deg // 64 and cnt <= 2 * c


def edges(rng):
    src, dst = [], []
    for i, deg in enumerate(DEGREES):
        v = 17 + 11 * i  # several in one group of 32 rows
        s = 10 + rng.choice(N - 11, deg, replace=False)  # nodes 0 to 9 stay without out-edges
        src.append(s + (s >= v))  # distinct sources, no self-loop
        dst.append(np.full(deg, v))
    # a sparse rest, so that mass returns to the sources above
    src.append(rng.integers(10, N, 2 * N))
    dst.append(rng.integers(0, N, 2 * N))
    return np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32)


@pytest.fixture(scope="module")
def case():
    import torch
    src, dst = edges(np.random.default_rng(3))
    g = gpr.graph_build(torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda(), N)
    ref = oracle.build_csc(N, src, dst)
    assert (ref.outdeg[:10] == 0).all()
    seeds = np.concatenate([[17 + 11 * 30, 17, 17 + 11, 0, 9], 1 + np.arange(60) * 541]).astype(np.int32)
    return torch, g, ref, seeds


def solve(torch, g, seeds, iters, dt, tol=0.0):
    x = torch.zeros((N, len(seeds)), dtype=torch.float32, device="cuda")
    res = gpr.ppr_batch([(g, seeds, 0.85, x)], max_iters=iters, tol=tol, dtype=dt)
    return x.cpu().numpy(), res[0]


@pytest.mark.gpu
@pytest.mark.parametrize("dt,err", [(gpr.FP32, 1e-5), (gpr.FP16, 1e-3), (gpr.BF16, 1e-3)])
@pytest.mark.parametrize("k", [1, 2, 4, 5, 16, 17, 64, 65])
def test_every_width_and_row_length(case, k, dt, err):
    torch, g, ref, seeds = case
    x, (it, res) = solve(torch, g, seeds[:k], 30, dt)
    assert (it == 30).all()
    for j in sorted({0, 1 % k, 3 % k, k - 1}):
        assert l1(x[:, j], oracle.ppr(ref, int(seeds[j]), 0.85, 30)[0]) <= err
    # the cluster schedule rounds otherwise, within twice the storage's error
    try:
        os.environ["GPR_PPR_CLUSTER"] = "4"
        y, (it2, res2) = solve(torch, g, seeds[:k], 30, dt)
    finally:
        os.environ.pop("GPR_PPR_CLUSTER", None)
    assert np.abs(x.astype(np.float64) - y).sum(0).max() <= 2 * err
    assert (it == it2).all() and np.abs(res - res2).max() <= 2 * err


@pytest.mark.gpu
@pytest.mark.parametrize("dt", [gpr.FP32, gpr.FP16, gpr.BF16])
def test_bits_do_not_depend_on_the_width(case, dt):
    torch, g, ref, seeds = case
    full, (_, r64) = solve(torch, g, seeds[:64], 25, dt)
    for k in (1, 3, 9, 40):
        part, (_, rk) = solve(torch, g, seeds[:k], 25, dt)
        assert (part == full[:, :k]).all() and (rk == r64[:k]).all()


@pytest.mark.gpu
def test_columns_that_stop_at_different_steps(case):
    torch, g, ref, seeds = case
    x, (it, res) = solve(torch, g, seeds[:7], 200, gpr.FP32, tol=1e-4)
    for j in range(7):
        xr, k_ref = oracle.ppr(ref, int(seeds[j]), 0.85, 200, 1e-4)
        assert abs(int(it[j]) - k_ref) <= 1 and 0.85 / 0.15 * res[j] <= 1e-4 * (1 + 1e-3)
        assert l1(x[:, j], oracle.ppr(ref, int(seeds[j]), 0.85, 300)[0]) <= 1e-4 + 1e-5


@pytest.mark.gpu
@pytest.mark.parametrize("k", [1, 3, 16, 64])
def test_bf16_rows_below_zero(k):
    # a cycle with a chord and a dangling node after node 4: as the front passes,
    # x[4] falls by a factor of a thousand in one step, the rounding of the sent
    # delta overshoots it, and the dangling mass is below zero at steps 12 (from
    # node 0) and 9 (from node 3).  A step's rounding moves at most 2^-9 of
    # ||x_k - x_{k-1}||_1 <= 2 (and of the rounding before), so 30 steps are
    # within 30 * 2.01 * 2^-9 of the exact ones
    import torch
    src, dst = np.array([0, 1, 2, 3, 4, 4, 3], np.int32), np.array([1, 2, 3, 4, 0, 5, 1], np.int32)
    g, ref = gpr.graph_build(src, dst, 6), oracle.build_csc(6, src, dst)
    seeds = np.resize(np.array([0, 3], np.int32), k)
    x = torch.zeros((6, k), dtype=torch.float32, device="cuda")
    gpr.ppr_batch([(g, seeds, 0.999, x)], max_iters=30, dtype=gpr.BF16)
    for j in range(min(k, 2)):
        assert l1(x[:, j].cpu().numpy(), oracle.ppr(ref, int(seeds[j]), 0.999, 30)[0]) <= 0.12


@pytest.mark.gpu
@pytest.mark.parametrize("k", [1, 4, 16, 64])
def test_hub_of_equal_contributions(k):
    # 130,000 nodes point at node 0, which points back: after two steps from node 0
    # its row sums as many equal numbers, 0.85 of the mass, in 508 chunks of 256 edges.
    # A slot rounds at most 8 times, the slots of a block twice, four blocks, the two
    # halves, 7 additions of an eight and 64 over the eights, half an ulp of 2^-24 each,
    # all the same way: 0.85 * 0.85 * 86 * 2^-25; the other roundings are 2.5e-7 together
    import torch
    n = 130_001
    o = np.arange(1, n, dtype=np.int32)
    z = np.zeros(n - 1, np.int32)
    src, dst = np.concatenate([o, z]), np.concatenate([z, o])
    g, ref = gpr.graph_build(src, dst, n), oracle.build_csc(n, src, dst)
    x = torch.zeros((n, k), dtype=torch.float32, device="cuda")
    gpr.ppr_batch([(g, np.zeros(k, np.int32), 0.85, x)], max_iters=2)
    want = oracle.ppr(ref, 0, 0.85, 2)[0]
    for j in {0, k - 1}:
        assert l1(x[:, j].cpu().numpy(), want) <= 0.85 * 0.85 * 86 * 2.0 ** -25 + 2.5e-7
