"""The default of the split-precision product on atoms of several row tiles: one or two
row tiles per B tile, whichever balances the SMs' lists.  9 x 9 lens-graded atoms of 240
unknowns leave half the SMs idle with two (1.4 times as long), 16 x 16 win with two."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("array,nrhs", [("graded 9 4", 16), ("square 10 4", 8), ("square 5 5", 24), ("square 16 4", 16)])
def test_default_is_the_faster_shape(array, nrhs):
    import torch
    from paper_2603_10586_gb300 import vie
    kind, n, nv = array.split()
    ctx = vie.Context(0)
    op = vie.Operator(ctx, workloads.square_array(int(n), int(nv)) if kind == "square" else
                      workloads.graded_array(int(n), int(nv), 9))
    op.compress(1e-4, vie.C64)
    x = torch.from_numpy(workloads.random_complex(op.n, 3, nrhs).T.astype(np.complex64).copy()).cuda()
    y = torch.empty_like(x)
    s = torch.cuda.Stream()

    def us():
        times = []
        for _ in range(6):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record(s)
            for _ in range(30):
                op.apply(x.data_ptr(), y.data_ptr(), nrhs, vie.BF16X3, 0, stream=s.cuda_stream)
            b.record(s)
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) / 30e-3)
        return min(times[1:])

    t = us()
    seen = []
    for _ in range(3):       # (a clock that moves between the two is measured again)
        shapes = []
        for v in (vie.VAR_TCGEN05_WS_BF16X3, vie.VAR_TCGEN05_WS2_BF16X3):
            op.tune(vie.BF16X3, nrhs, force=v)
            shapes.append(us())
        seen.append(shapes)
        if t < 1.06 * min(shapes):
            break
    else:
        raise AssertionError((t, seen))
    op.close()
    ctx.close()
