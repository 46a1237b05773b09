"""Field read-outs whose partial sums take several passes, in a context whose
memory holds the output once and not twice.  The passes end inside the points or
directions; their ends are compared with small calls (the same sums in the same
order: one atom is one chunk)."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,nrhs,npts,budget", [("near", 4, 1_000_003, 300), ("far", 64, 40_001, 200)])
def test_output_is_held_once(mode, nrhs, npts, budget):
    from paper_2603_10586_gb300 import vie
    ctx = vie.Context(0, hbm_budget=budget << 20)
    op = vie.Operator(ctx, workloads.single_cube(0.2, 1))
    I = workloads.random_complex(op.n, 4, nrhs)
    p = np.random.default_rng(5).uniform(0.5, 2.0, (npts, 3))
    if mode == "far":
        p /= np.linalg.norm(p, axis=1, keepdims=True)
    read = op.near_field if mode == "near" else op.far_field
    out = read(I, p)
    per = (32 << 20) // (48 * nrhs)      # points of one pass
    for at in (0, per - 40, 2 * per - 40, npts - 80):
        want = read(I, p[at:at + 80])
        assert np.abs(out[:, at:at + 80] - want).max() <= 1e-13 * np.abs(want).max()
    op.close()
    ctx.close()


@pytest.mark.parametrize("budget", [22, 26])
def test_passes_fit_a_small_budget(budget):
    # 18 MB of amplitudes in a context of 22 and 26 MB: shorter passes, not VIE_ERR_OOM
    from paper_2603_10586_gb300 import vie
    rng = np.random.default_rng(3)
    p = rng.uniform(0.5, 2.0, (6000, 3)) + [0, 0, 3.0]
    d = p / np.linalg.norm(p, axis=1, keepdims=True)
    out = []
    for mb in (0, budget):
        ctx = vie.Context(0, hbm_budget=mb << 20)
        op = vie.Operator(ctx, workloads.vogel_gold(40, 2))
        I = workloads.random_complex(op.n, 4, 64)
        kh, pol = workloads.random_directions(64, 2)
        out.append((op.far_field(I, d), op.near_field(I, p), op.sigma(I, kh, pol)))
        op.close()
        ctx.close()
    for a, b in zip(*out):
        # float64 sums of ~1,400 terms in another order
        assert np.abs(a - b).max() <= 1e-11 * np.abs(a).max()
