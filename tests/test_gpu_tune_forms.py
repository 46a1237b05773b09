"""The autotuner chooses between the register tiles and the per-block kernels of two,
four and eight right-hand sides, not between three names of one kernel."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _launches(vie, f):
    import torch
    n = vie.kernel_launches()
    f()
    torch.cuda.synchronize()
    return vie.kernel_launches() - n


@pytest.mark.parametrize("nrhs", [2, 5])
def test_tuner_times_both_forms(nrhs):
    import torch
    from paper_2603_10586_gb300 import vie
    ctx = vie.Context(0)
    op = vie.Operator(ctx, workloads.square_array(6, 3))
    op.compress(1e-4, vie.C64)
    X = torch.from_numpy(workloads.random_complex(op.n, 2, nrhs).T.astype(np.complex64).copy()).cuda()
    Y = torch.empty_like(X)
    apply = lambda: op.apply(X.data_ptr(), Y.data_ptr(), nrhs, vie.C64, 0)  # noqa: E731
    apply()
    tiles = _launches(vie, apply) - 1            # without the self blocks' product
    want = Y.cpu().numpy()
    op.tune(vie.C64, nrhs, force=vie.VAR_SIMT_R1)
    one = _launches(vie, apply) - 1
    blocks = 2                                   # phase 1 and phase 2 of any group size
    assert tiles > blocks
    # four passes each of R1, of R2, R4 and R8 as per-block kernels, and of the tiles
    assert _launches(vie, lambda: op.tune(vie.C64, nrhs)) == 4 * (one + 3 * blocks + tiles)
    apply()
    torch.cuda.synchronize()
    y = Y.cpu().numpy()
    assert np.linalg.norm(y - want) < 1e-6 * np.linalg.norm(want)
    op.close()
    ctx.close()
