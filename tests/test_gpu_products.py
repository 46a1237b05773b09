"""Register-tile products at the edges of their tiles: rows, columns and K ranges
that end inside a tile, single copies and groups of more than 64, segments of a
long row, all arithmetics.  Reference: the exported factors and self blocks
multiplied out in float64.  A float32 sum of K products is off by at most
K 2^-24 of its terms' magnitude and about sqrt(K) 2^-24 of its size: with K <=
1500 the bound of 1e-5 of the result's norm leaves room for cancellation; the
float64-accurate products carry at least 2^-46."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _reference(op, g, x, fused):
    far = np.zeros_like(x)
    n = op.np
    for b in op.far_blocks():
        t = np.concatenate([np.arange(a * n, (a + 1) * n) for a in b["tatoms"]])
        s = np.concatenate([np.arange(a * n, (a + 1) * n) for a in b["satoms"]])
        far[:, t] += x[:, s] @ b["R"].T @ b["Q"].T
    out = np.zeros_like(x)
    for t in range(len(g.sides)):
        M = op.export_block(2 if fused else 0, t)
        for a in np.flatnonzero(g.types == t):
            r = slice(a * n, (a + 1) * n)
            out[:, r] = x[:, r] + far[:, r] @ M.T if fused else x[:, r] @ M.T + far[:, r]
    return out


# (array, tolerance of the compression, precision, columns)
CASES = [("square 3 1", 1e-4, "C64", 1), ("square 9 2", 1e-4, "C64", 1), ("square 9 2", 1e-4, "C64", 7),
         ("graded 6 3", 1e-3, "C64", 2), ("spiral 20 2", 1e-4, "C64", 5), ("square 8 5", 1e-2, "C64", 3),
         ("square 12 2", 1e-4, "C64_ACC64", 3), ("graded 5 3", 1e-4, "C64_ACC64", 9), ("square 4 4", 1e-5, "C64_ACC64", 1),
         ("square 9 2", 1e-5, "C128", 2), ("graded 4 3", 1e-6, "C128", 5)]


@pytest.mark.parametrize("array,tol,precision,nrhs", CASES)
def test_apply(array, tol, precision, nrhs):
    import torch
    from paper_2603_10586_gb300 import vie
    kind, size, nv = array.split()
    g = (workloads.square_array(int(size), int(nv)) if kind == "square" else
         workloads.graded_array(int(size), int(nv), 1) if kind == "graded" else workloads.vogel_gold(int(size), int(nv)))
    prec = getattr(vie, precision)
    ctx = vie.Context(0)
    op = vie.Operator(ctx, g)
    op.compress(tol, vie.C128 if precision == "C128" else vie.C64)
    x = workloads.random_complex(op.n, 5, nrhs).T.copy()
    X = torch.from_numpy(x.astype(np.complex64 if precision == "C64" else np.complex128)).cuda()
    Y = torch.empty_like(X)
    for fused in (False, True):
        op.apply(X.data_ptr(), Y.data_ptr(), nrhs, prec, vie.FUSE_PRECOND if fused else 0)
        torch.cuda.synchronize()
        ref = _reference(op, g, X.cpu().numpy().astype(np.complex128), fused)
        err = np.linalg.norm(Y.cpu().numpy() - ref) / np.linalg.norm(ref)
        assert err < (1e-5 if precision == "C64" else 1e-12), (fused, err)
    op.close()
    ctx.close()


# atoms of 6 to 450 unknowns (not whole chunks of 8, one to four row tiles), ragged
# ranks and column counts, one and two 64-column passes, with and without copies.  A
# split operand keeps 16 bits: 2^-16 per factor and value, 5e-5 of the norm in all.
@pytest.mark.parametrize("array,tol,nrhs", [("square 3 1", 1e-4, 8), ("square 8 1", 1e-2, 17), ("spiral 20 2", 1e-4, 9),
                                            ("graded 5 3", 1e-4, 33), ("square 6 5", 1e-3, 12), ("square 5 3", 1e-5, 65)])
@pytest.mark.parametrize("variant", ["VAR_TCGEN05_WS_BF16X3", "VAR_TCGEN05_WS2_BF16X3"])
def test_tensor_core_apply(array, tol, nrhs, variant):
    import torch
    from paper_2603_10586_gb300 import vie
    kind, size, nv = array.split()
    g = (workloads.square_array(int(size), int(nv)) if kind == "square" else
         workloads.graded_array(int(size), int(nv), 1) if kind == "graded" else workloads.vogel_gold(int(size), int(nv)))
    ctx = vie.Context(0)
    op = vie.Operator(ctx, g)
    op.compress(tol, vie.C64)
    op.tune(vie.BF16X3, nrhs, force=getattr(vie, variant))
    X = torch.from_numpy(workloads.random_complex(op.n, 8, nrhs).T.astype(np.complex64).copy()).cuda()
    Y = torch.empty_like(X)
    op.apply(X.data_ptr(), Y.data_ptr(), nrhs, vie.BF16X3, 0)
    torch.cuda.synchronize()
    ref = _reference(op, g, X.cpu().numpy().astype(np.complex128), False)
    err = np.linalg.norm(Y.cpu().numpy() - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert err.max() < 5e-5
    op.close()
    ctx.close()


@pytest.mark.parametrize("ns,nv,nrhs", [(1, 1, 1), (2, 3, 1), (3, 4, 5), (7, 2, 11), (16, 3, 9), (12, 4, 33)])
@pytest.mark.parametrize("precision", ["C64", "C128"])
def test_precond(ns, nv, nrhs, precision):
    import torch
    from paper_2603_10586_gb300 import vie
    g = workloads.graded_array(ns, nv, 2)
    ctx = vie.Context(0)
    op = vie.Operator(ctx, g)
    x = workloads.random_complex(op.n, 6, nrhs).T.copy()
    X = torch.from_numpy(x.astype(np.complex64 if precision == "C64" else np.complex128)).cuda()
    Y = torch.empty_like(X)
    op.precond(X.data_ptr(), Y.data_ptr(), nrhs, getattr(vie, precision))
    torch.cuda.synchronize()
    x = X.cpu().numpy().astype(np.complex128).reshape(nrhs, g.n_atoms, op.np)
    ref = np.zeros_like(x)
    for t in range(len(g.sides)):
        inv = op.export_block(2, t)
        ref[:, g.types == t] = x[:, g.types == t] @ inv.T
    err = np.linalg.norm(Y.cpu().numpy() - ref.reshape(nrhs, -1)) / np.linalg.norm(ref)
    assert err < (1e-5 if precision == "C64" else 1e-13)
    op.close()
    ctx.close()


# short items (16 rows of R, 32 of Q in complex128; 32 and 64 where shared factors
# leave few items) and long ones (64 and 256) with one to two column tiles
@pytest.mark.parametrize("array,tol,precision,nrhs", [
    ("square 5 3", 1e-4, "C128", 1), ("spiral 12 2", 1e-3, "C128", 4), ("square 3 4", 1e-6, "C128", 9),
    ("square 7 3", 1e-5, "C64", 1), ("square 5 4", 1e-3, "C64", 6), ("spiral 25 3", 1e-5, "C64", 9),
    ("square 18 3", 1e-4, "C64", 1), ("square 6 3", 1e-2, "C64_ACC64", 2)])
def test_apply_item_rows(array, tol, precision, nrhs):
    test_apply(array, tol, precision, nrhs)
