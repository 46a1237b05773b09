"""The explicit inverse of a self block from the smallest block to one whose
columns no longer fit in shared memory (1, 2, 5 and 8 voxels per edge: 6, 36,
450 and 1,728 unknowns), for two types at once."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nv", [1, 2, 5, 8])
def test_inverse(nv):
    from paper_2603_10586_gb300 import vie
    g = workloads.two_cubes(0.6, nv=nv)
    g.types, g.sides = np.array([0, 1], np.int32), np.array([0.2, 0.15])
    g.nvs, g.eps = np.array([nv, nv], np.int32), np.array([12.0, 6.0 - 0.5j], complex)
    ctx = vie.Context(0)
    op = vie.Operator(ctx, g)
    for t in range(2):
        Z, inv = op.export_block(0, t), op.export_block(2, t)
        n = len(Z)
        # backward stable up to growth: n eps cond, cond of these blocks below 1e4
        bound = 1e-12 * n
        assert np.abs(inv @ Z - np.eye(n)).max() < bound
        assert np.abs(Z @ inv - np.eye(n)).max() < bound
    op.close()
    ctx.close()
