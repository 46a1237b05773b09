"""Right-hand sides, far field, near field and cross sections against the oracle
where the column, direction and atom groups of the kernels end: one and several
voxels per edge, several atom types (one of them unused), 1 to 6 columns, 1 to
300 directions.  Both sides are float64 evaluations of the same 3-point rule, so
they differ by summation order only: 1e-12 of the largest entry."""
import numpy as np
import pytest

import workloads
from oracle import assembly as A
from oracle import fields as F
from oracle import problem_from_geometry

pytestmark = pytest.mark.gpu
TOL = 1e-12


def _case(kind):
    if kind == "one":
        return workloads.single_cube(0.2, 1)
    if kind == "two":
        return workloads.two_cubes(0.7, nv=2)
    if kind == "graded":   # three types
        g = workloads.graded_array(3, 2, seed=3)
        g.types = np.array([0, 1, 2, 0, 1, 2, 2, 1, 0], np.int32)
        return g
    g = workloads.square_array(3, 3)   # the second of two types has no atom
    g.sides, g.nvs, g.eps = np.array([0.2, 0.1]), np.array([3, 3], np.int32), np.array([12.0, 5.0], complex)
    return g


def _close(got, want):
    assert np.abs(got - want).max() <= TOL * np.abs(want).max()


@pytest.mark.parametrize("kind,nrhs,ndirs", [("one", 1, 1), ("two", 5, 3), ("graded", 4, 300), ("spare", 6, 17)])
def test_plane_waves_and_fields(kind, nrhs, ndirs):
    import torch
    from paper_2603_10586_gb300 import vie
    g = _case(kind)
    ctx = vie.Context(0)
    op = vie.Operator(ctx, g)
    P = problem_from_geometry(g)
    kh, pol = workloads.random_directions(nrhs, 7, max_deg=80.0)
    b = torch.zeros((nrhs, op.n), dtype=torch.complex128, device="cuda")
    op.rhs(kh, pol, b.data_ptr())
    want = np.stack([A.rhs(P, kh[c], pol[c]) for c in range(nrhs)])
    _close(b.cpu().numpy(), want)
    I = workloads.random_complex(op.n, 11, nrhs)
    rng = np.random.default_rng(2)
    d = rng.standard_normal((ndirs, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    far, sig = op.far_field(I, d), op.sigma(I, kh, pol)
    pts = np.concatenate([rng.uniform(-0.8, 0.8, (3, 2)), rng.uniform(0.3, 2.0, (3, 1))], 1)
    near = op.near_field(I, pts)
    for c in range(nrhs):
        _close(far[c], F.far_field(P, I[:, c], d))
        _close(near[c], F.near_field(P, I[:, c], pts))
        assert abs(sig[c, 1] - F.sigma_sca(P, I[:, c])) <= TOL * sig[c, 1]
        v0 = want[c] / (1j * P.k)
        # the extinction may cancel: compare at the scale of its terms
        assert abs(sig[c, 0] - F.sigma_ext(I[:, c], v0)) <= TOL * np.abs(I[:, c]) @ np.abs(v0)
    op.close()
    ctx.close()
