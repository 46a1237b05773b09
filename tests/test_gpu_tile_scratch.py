"""The register tiles' scratch is optional: a call that gets none of it, or half of it,
runs the per-block kernels, and a call that is short of memory gets back what an
earlier one kept.  Also calls of more columns than one pass takes (1,024)."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _open(budget=0):
    from paper_2603_10586_gb300 import vie
    ctx = vie.Context(0, hbm_budget=budget << 20)
    op = vie.Operator(ctx, workloads.square_array(12, 2))
    op.compress(1e-4, vie.C64)
    return vie, ctx, op


def _apply(vie, op, x, precision):
    import torch
    X = torch.from_numpy(x).cuda()
    Y = torch.empty_like(X)
    op.apply(X.data_ptr(), Y.data_ptr(), len(x), precision, 0)
    torch.cuda.synchronize()
    return Y.cpu().numpy()


def _worst(a, b):
    return (np.linalg.norm(a - b, axis=1) / np.linalg.norm(b, axis=1)).max()


def test_short_of_scratch():
    # 64 columns of 16 bytes: 242 MB of partial products, 220 MB of segmented t;
    # the per-block kernels' t takes 183 MB.  Both add the same float64-accurate
    # products in another order.
    x = workloads.random_complex(12 * 12 * 36, 3, 64).T.copy()
    vie, ctx, op = _open()
    want = _apply(vie, op, x, vie.C64_ACC64)
    op.close()
    ctx.close()
    for budget in (320, 420, 480, 700):
        vie, ctx, op = _open(budget)
        for _ in range(2):
            assert _worst(_apply(vie, op, x, vie.C64_ACC64), want) < 1e-12
        op.close()
        ctx.close()


def test_solve_after_a_wide_apply():
    # the apply keeps 460 MB; the solve needs 330 MB of Krylov vectors and 230 MB besides
    x = workloads.random_complex(12 * 12 * 36, 3, 64).T.copy()
    kh, pol = workloads.random_directions(64, 5)
    sol = []
    for budget, wide in ((0, False), (800, True)):
        vie, ctx, op = _open(budget)
        if wide:
            _apply(vie, op, x, vie.C64_ACC64)
        I, st, status = op.solve(kh, pol, tol=1e-6)
        assert status == vie.VIE_OK and st["residual"] <= 1e-6
        sol.append(I.T.copy())
        op.close()
        ctx.close()
    # two solutions to a residual of 1e-6: their difference stays near it
    assert _worst(sol[1], sol[0]) < 1e-5


@pytest.mark.parametrize("precision,tol", [("C64", 1e-5), ("C64_ACC64", 1e-12)])
def test_more_columns_than_a_pass(precision, tol):
    from paper_2603_10586_gb300 import vie
    ctx = vie.Context(0)
    op = vie.Operator(ctx, workloads.square_array(3, 1))
    op.compress(1e-4, vie.C64)
    x = workloads.random_complex(op.n, 7, 1100).T.astype(np.complex64 if precision == "C64" else np.complex128)
    y = _apply(vie, op, np.ascontiguousarray(x), getattr(vie, precision))
    # the dense matrix of the operator from its exported blocks, in float64
    Z = np.zeros((op.n, op.n), complex)
    n = op.np
    for b in op.far_blocks():
        t = np.concatenate([np.arange(a * n, (a + 1) * n) for a in b["tatoms"]])
        s = np.concatenate([np.arange(a * n, (a + 1) * n) for a in b["satoms"]])
        Z[np.ix_(t, s)] += b["Q"] @ b["R"]
    for a in range(9):
        Z[a * n:(a + 1) * n, a * n:(a + 1) * n] += op.export_block(0, 0)
    assert _worst(y, x.astype(np.complex128) @ Z.T) < tol
    op.close()
    ctx.close()
