"""The self-block product (preconditioner) where its tiles lost time: blocks of one voxel per
edge, which leave most of a 64-row tile empty, and complex128 columns that left most SMs
waiting for the last of their tiles."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _precond(g, nrhs, precision):
    """(us per call on the device, worst column's error against the exported inverses)"""
    import torch
    from paper_2603_10586_gb300 import vie
    ctx = vie.Context(0)
    op = vie.Operator(ctx, g)
    wide = precision == "C128"
    x = workloads.random_complex(op.n, 6, nrhs).T.astype(np.complex128 if wide else np.complex64).copy()
    X = torch.from_numpy(x).cuda()
    Y = torch.empty_like(X)
    call = lambda: op.precond(X.data_ptr(), Y.data_ptr(), nrhs, getattr(vie, precision))  # noqa: E731
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        call()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        for _ in range(20):
            call()
    times = []
    for _ in range(6):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        graph.replay()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b) * 50.0)
    v = x.astype(complex).reshape(nrhs, g.n_atoms, op.np)
    ref = np.zeros_like(v)
    for t in range(len(g.sides)):
        ref[:, g.types == t] = v[:, g.types == t] @ op.export_block(2, t).T
    ref = ref.reshape(nrhs, -1)
    err = (np.linalg.norm(Y.cpu().numpy() - ref, axis=1) / np.linalg.norm(ref, axis=1)).max()
    op.close()
    ctx.close()
    return min(times), err


# six products per sum: float32 rounding of a few terms, float64 likewise
@pytest.mark.parametrize("ns,nrhs", [(1, 1), (3, 5), (11, 3), (24, 33)])
@pytest.mark.parametrize("precision,tol", [("C64", 1e-6), ("C128", 1e-14)])
def test_one_voxel_blocks(ns, nrhs, precision, tol):
    assert _precond(workloads.graded_array(ns, 1, 2), nrhs, precision)[1] < tol


def _below(most, g, one, other, precision):
    """us(one columns) <= most us(other columns), in the best of three pairs."""
    ratios = []
    for _ in range(3):
        ratios.append(_precond(g, one, precision)[0] / _precond(g, other, precision)[0])
        if ratios[-1] < most:
            return
    raise AssertionError(ratios)


def test_one_voxel_blocks_time():
    # 24 x 24 atoms: 33 columns move 0.9 MB; one column is a launch (3.3 us).  64-row tiles: 2.5 times it
    _below(2.2, workloads.square_array(24, 1), 33, 1, "C64")


@pytest.mark.parametrize("ns,nv,nrhs", [(9, 4, 33), (9, 4, 24), (7, 5, 64), (16, 4, 16), (8, 3, 33)])
def test_float64_columns(ns, nv, nrhs):
    # sums of up to 450 products in float64
    assert _precond(workloads.square_array(ns, nv), nrhs, "C128")[1] < 1e-13


def test_float64_columns_time():
    # 33 columns of 81 atoms of 240 unknowns as 336 tiles: three on some SMs, 2.2 on average
    _below(1.03 * 33 / 24, workloads.square_array(9, 4), 33, 24, "C128")
