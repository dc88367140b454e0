"""Which schedule ppr_batch runs: what the tuner says it keeps is what later calls
run, and the environment variable forces either, whatever was tuned."""
import os

import numpy as np
import pytest

import paper_1606_07550_gb300 as gpr
from test_ppr_steps import N, case, solve  # noqa: F401 (case is a fixture)

pytestmark = pytest.mark.gpu

STEPS = 25


def launches(f):
    before = gpr.lib().gpr_kernel_launches()
    out = f()
    return gpr.lib().gpr_kernel_launches() - before, out


@pytest.fixture
def force():
    def set_to(shape):
        os.environ["GPR_PPR_CLUSTER"] = shape
    yield set_to
    os.environ.pop("GPR_PPR_CLUSTER", None)


@pytest.mark.parametrize("dt", [gpr.FP32, gpr.FP16, gpr.BF16])
def test_tuner_says_what_later_calls_run(case, dt):
    torch, g, ref, seeds = case
    x = torch.zeros((N, 64), dtype=torch.float32, device="cuda")
    (r,) = gpr.ppr_tune([(g, seeds[:64], 0.85, x)], dtype=dt, trial_steps=5)
    assert r["ms_steps"] > 0 and r["cluster"] in (1, 2, 4, 8)
    assert r["kept"] == (0 if r["ms_steps"] < r["ms"] else r["cluster"])
    count, _ = launches(lambda: solve(torch, g, seeds[:64], STEPS, dt))
    assert (count > STEPS) == (r["kept"] == 0)  # a launch a step or more, or one launch in all


@pytest.mark.parametrize("dt", [gpr.FP32, gpr.FP16, gpr.BF16])
def test_forced_schedules_and_their_bits(case, force, dt):
    torch, g, ref, seeds = case
    force("4")
    count, _ = launches(lambda: solve(torch, g, seeds[:64], STEPS, dt))
    assert count == 1
    # step by step: the same bits at every width, whatever the tuner keeps
    force("0")
    count, (full, (_, r64)) = launches(lambda: solve(torch, g, seeds[:64], STEPS, dt))
    assert count > STEPS
    for k in (1, 3, 9, 40):
        part, (_, rk) = solve(torch, g, seeds[:k], STEPS, dt)
        assert (part == full[:, :k]).all() and (rk == r64[:k]).all()


def test_workspace_of_a_batch_is_bounded(force):
    # 30 jobs of 2^20 nodes, 64 columns in BF16, are 22.5 GB of state: three waves
    import ctypes
    import torch
    cu = ctypes.CDLL("libcuda.so.1")
    pool, dev, used = ctypes.c_void_p(), ctypes.c_int(), ctypes.c_uint64()
    used_now, used_high = 7, 8  # CU_MEMPOOL_ATTR_USED_MEM_CURRENT, _HIGH

    def pool_use(attr):
        assert cu.cuMemPoolGetAttribute(pool, attr, ctypes.byref(used)) == 0
        return used.value

    n, k, jobs = 1 << 20, 64, 30
    gen = torch.Generator(device="cuda").manual_seed(2)
    src, dst = (torch.randint(0, n, (n,), dtype=torch.int32, device="cuda", generator=gen) for _ in range(2))
    g = gpr.graph_build(src, dst, n)
    seeds = np.arange(k, dtype=np.int32) * 977
    x = [torch.zeros((n, k), dtype=torch.float32, device="cuda") for _ in range(jobs)]
    assert cu.cuCtxGetDevice(ctypes.byref(dev)) == 0 and cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), dev) == 0
    force("0")
    gpr.ppr_batch([(g, seeds, 0.85, x[0])], max_iters=3, dtype=gpr.BF16)
    alone = x[0].clone()
    before = pool_use(used_now)
    zero = ctypes.c_uint64(0)
    assert cu.cuMemPoolSetAttribute(pool, used_high, ctypes.byref(zero)) == 0
    gpr.ppr_batch([(g, seeds, 0.85, o) for o in x], max_iters=3, dtype=gpr.BF16)
    assert pool_use(used_high) - before <= (8 << 30) + (64 << 20)  # and records, items, piece bounds
    for o in x:
        assert torch.equal(o, alone)
