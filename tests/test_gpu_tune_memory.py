"""What tuning leaves on the GPU: the planes of the shared-storage tensor-core kernels, not
those of the per-block ones (3.2 GB here) unless they were chosen."""
import pytest

import workloads

pytestmark = pytest.mark.gpu


def test_tuning_keeps_one_set_of_planes():
    import torch
    from paper_2603_10586_gb300 import vie
    ctx = vie.Context(0)
    op = vie.Operator(ctx, workloads.square_array(16, 4))
    op.compress(1e-4, vie.C64)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    r = op.tune(vie.BF16X3, 16)
    torch.cuda.synchronize()
    assert r["variant"] != vie.VAR_TCGEN05_PACKED_BF16X3
    assert vie.VAR_TCGEN05_PACKED_BF16X3 in r["ms"]
    assert free - torch.cuda.mem_get_info()[0] < 1.5e9
    op.close()
    ctx.close()


def test_tuning_under_a_budget():
    from paper_2603_10586_gb300 import vie
    # room for the operator and its shared planes, not for the planes per block: 7 runs as 6
    ctx = vie.Context(0, hbm_budget=3000 << 20)
    op = vie.Operator(ctx, workloads.square_array(16, 4))
    op.compress(1e-4, vie.C64)
    r = op.tune(vie.BF16X3, 64)
    assert len(r["ms"]) == 9
    op.close()
    ctx.close()
