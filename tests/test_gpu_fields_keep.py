"""Workspaces that a field read-out keeps do not take a later call's memory: under the
smallest budget (in steps of 20 MB) that holds a solve, the same solve after a read-out."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _solve(budget_mb, read_out):
    """The solve's currents, None when the budget does not hold it."""
    from paper_2603_10586_gb300 import vie
    ctx = vie.Context(0, hbm_budget=budget_mb << 20)
    kh, pol = workloads.random_directions(48, 5)
    I = None
    try:
        op = vie.Operator(ctx, workloads.square_array(12, 2))
        op.compress(1e-4, vie.C64)
        if read_out:
            # 48 currents in 24,000 directions: 55 MB of amplitudes, 32 MB each of tables and sums
            d = np.random.default_rng(1).standard_normal((24000, 3))
            d /= np.linalg.norm(d, axis=1, keepdims=True)
            op.far_field(workloads.random_complex(op.n, 2, 48), d)
        I, st, status = op.solve(kh, pol, tol=1e-6)
        assert status == vie.VIE_OK
        op.close()
    except vie.VieError as e:
        assert e.status == vie.VIE_ERR_OOM
    ctx.close()
    return I


def test_solve_after_a_read_out():
    for budget in range(300, 900, 20):
        want = _solve(budget, False)
        if want is not None:
            break
    got = _solve(budget, True)
    assert got is not None
    # two solutions to a residual of 1e-6
    assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)
