"""What a server's slot keeps between requests: its pool of temporaries goes back with
the request's footprint, so that other requests can be promised the memory."""
import time

import pytest

import workloads

pytestmark = pytest.mark.gpu


def _free_mb():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0] / 2**20


def _serve(srv, vie, n):
    t = srv.submit(workloads.square_array(n, 3), *workloads.random_directions(2, 1))
    r, end = None, time.time() + 120
    while r is None and time.time() < end:
        r = srv.poll(t, timeout_ms=1000)
    assert r is not None and r["status"] == vie.VIE_OK


def test_slot_gives_its_pool_back():
    from paper_2603_10586_gb300 import vie
    ctx = vie.Context(0)
    srv = vie.Server(ctx, max_inflight=1, tol=1e-4)
    _serve(srv, vie, 12)         # kernels and cuBLAS loaded, handle and workspace made
    idle = _free_mb()
    srv.stop()
    closed = _free_mb()
    # a context that compressed the same operator holds a stream, a cuBLAS handle and its pool
    ctx2 = vie.Context(0)
    op = vie.Operator(ctx2, workloads.square_array(12, 3))
    op.compress(1e-4, vie.C64)
    op.close()
    with_pool = _free_mb()
    ctx2.close()
    after = _free_mb()
    assert abs(after - closed) <= 8
    assert closed - idle < after - with_pool - 64
    ctx.close()
