"""A server's tick that fails on the host (no memory for its items): the running
requests fail, and nothing of them is left for the requests after them."""
import os

import numpy as np
import pytest

import gen
import oracle
import paper_1606_07550_gb300 as gpr

from gpu_util import l1

pytestmark = pytest.mark.gpu


def wait(srv, ticket):
    for _ in range(600):
        r = srv.poll(ticket, 100_000)
        if r is not None:
            return r
    raise AssertionError("request did not finish")


def result(torch, srv, ticket, r):
    out = torch.empty(r.n * r.num_seeds, device="cuda")
    srv.fetch(ticket, out)
    return out.cpu().numpy().reshape(r.n, r.num_seeds)


@pytest.mark.parametrize("dt,err", [(gpr.FP32, 1e-5), (gpr.BF16, 1e-3)])
def test_requests_after_a_failed_tick(dt, err):
    import torch
    src, dst = gen.rmat_coo(3000, 40_000, seed=61)
    g, ref = gpr.graph_build(src, dst, 3000), oracle.build_csc(3000, src, dst)
    pool_bytes = g.info().device_bytes
    new = dict(graph_id=0, seeds=[5, 2999], damping=0.83, max_iters=60, dtype=dt)
    with_server = gpr.Server([g], budget_bytes=4 << 30)
    t = with_server.submit(**new)
    want = result(torch, with_server, t, wait(with_server, t))
    with_server.close()
    os.environ["GPR_INJECT_TICK_FAILURE"] = "3"  # after two ticks of eight steps
    try:
        srv = gpr.Server([g], budget_bytes=4 << 30, steps_per_tick=8)
    finally:
        os.environ.pop("GPR_INJECT_TICK_FAILURE", None)
    # would take its 40 columns' 40 steps to the end while the next request runs
    old = srv.submit(0, list(range(40)), max_iters=40, dtype=dt)
    assert wait(srv, old).status == gpr.ECUDA
    st = srv.stats()
    assert st["failed"] == 1 and st["active_columns"] == 0
    assert st["device_bytes_in_use"] == pool_bytes + 3000 * 40 * 4  # the failed request's result, until released
    srv.release(old)
    tickets = [srv.submit(**new) for _ in range(3)]  # one of them where the old result was
    for t in tickets:
        r = wait(srv, t)
        assert r.status == gpr.OK and r.iters_max == 60
        x = result(torch, srv, t, r)
        assert (x == want).all()
        assert l1(x[:, 0], oracle.ppr(ref, 5, 0.83, 60)[0]) <= err
        srv.release(t)
    st = srv.stats()
    assert st["completed"] == 3 and st["failed"] == 1 and st["device_bytes_in_use"] == pool_bytes
    srv.close()


def test_fetch_to_device_memory_waits_for_its_copy():
    # the copy goes behind what the default stream holds, here about a second of
    # waiting: after it the result may be released and its memory used again
    import time
    import torch
    src, dst = gen.rmat_coo(3000, 40_000, seed=61)
    g = gpr.graph_build(src, dst, 3000)
    srv = gpr.Server([g], budget_bytes=4 << 30)
    t = srv.submit(0, [5], max_iters=20)
    r = wait(srv, t)
    out = torch.zeros(r.n, device="cuda")
    torch.cuda.synchronize()
    start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    start.record()
    torch.cuda._sleep(1_000_000_000)
    end.record()
    t0 = time.perf_counter()
    srv.fetch(t, out)
    waited = time.perf_counter() - t0
    assert end.query() and waited >= 0.5e-3 * start.elapsed_time(end)
    srv.release(t)
    srv.close()
