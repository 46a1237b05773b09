"""Two to five atoms: up to four columns go through the two per-block kernels and the
self-block product, more through the register tiles."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("atoms,nrhs,blocks", [(2, 1, True), (3, 4, True), (4, 4, True), (5, 1, True),
                                               (5, 2, False), (4, 5, False), (6, 1, False)])
@pytest.mark.parametrize("nv", [1, 3])
def test_launches(atoms, nrhs, blocks, nv):
    import torch
    from paper_2603_10586_gb300 import vie
    ctx = vie.Context(0)
    op = vie.Operator(ctx, workloads.vogel_gold(atoms, nv))
    op.compress(1e-4, vie.C64)
    x = workloads.random_complex(op.n, 5, nrhs).T.astype(np.complex64).copy()
    X = torch.from_numpy(x).cuda()
    Y = torch.empty_like(X)
    n = vie.kernel_launches()
    op.apply(X.data_ptr(), Y.data_ptr(), nrhs, vie.C64, 0)
    torch.cuda.synchronize()
    assert (vie.kernel_launches() - n == 3) == blocks
    ref = np.zeros(x.shape, complex)
    p = op.np
    for b in op.far_blocks():
        t = np.concatenate([np.arange(a * p, (a + 1) * p) for a in b["tatoms"]])
        s = np.concatenate([np.arange(a * p, (a + 1) * p) for a in b["satoms"]])
        ref[:, t] += x[:, s] @ b["R"].T @ b["Q"].T
    M = op.export_block(0, 0)
    for a in range(atoms):
        r = slice(a * p, (a + 1) * p)
        ref[:, r] += x[:, r] @ M.T
    # float32 sums of a few hundred products
    assert (np.linalg.norm(Y.cpu().numpy() - ref, axis=1) / np.linalg.norm(ref, axis=1)).max() < 1e-5
    op.close()
    ctx.close()


def test_grouped_kernels_keep_a_columns_order():
    # the per-block kernels of 2, 4 and 8 right-hand sides sum every column alike
    import torch
    from paper_2603_10586_gb300 import vie
    ctx = vie.Context(0)
    op = vie.Operator(ctx, workloads.vogel_gold(4, 3))
    op.compress(1e-5, vie.C64)
    X = torch.from_numpy(workloads.random_complex(op.n, 5, 4).T.astype(np.complex64).copy()).cuda()
    out = []
    for v in (vie.VAR_SIMT_R2, vie.VAR_SIMT_R4, vie.VAR_SIMT_R8):
        op.tune(vie.C64, 4, force=v)
        Y = torch.zeros_like(X)
        op.apply(X.data_ptr(), Y.data_ptr(), 4, vie.C64, vie.FUSE_PRECOND)
        torch.cuda.synchronize()
        out.append(Y.cpu().numpy())
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[1], out[2])
    op.close()
    ctx.close()
