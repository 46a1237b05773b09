"""The shared-factor apply, set by the caller, runs inside a solve's graphs as it does
launched from the host, whatever the default would be."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def test_shared_variant_inside_graphs():
    from paper_2603_10586_gb300 import vie
    ctx = vie.Context(0)
    op = vie.Operator(ctx, workloads.vogel_gold(250, nv=1))   # no shared factors: the rule takes the per-block kernels
    op.compress(1e-4, vie.C64)
    kh, pol = workloads.random_directions(1, 3)
    op.tune(vie.C64, 1, force=vie.VAR_SIMT_SHARED)
    Ig, _, sg = op.solve(kh, pol, tol=1e-6, restart=20, launch=0)
    Ih, _, sh = op.solve(kh, pol, tol=1e-6, restart=20, launch=1)
    assert sg == sh == vie.VIE_OK and np.array_equal(Ig, Ih)
    op.close()
    ctx.close()
