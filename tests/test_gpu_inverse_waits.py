"""The self-block inverse, whose CTAs wait for one another at bounded barriers: a grid
that gives up (a wait limit of zero cycles) is run again as one CTA, with the same
bits, and two contexts that invert at the same time, with blocks so large that an SM
holds one CTA, both finish."""
import threading

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _inverse(g, out, i):
    from paper_2603_10586_gb300 import vie
    ctx = vie.Context(0)
    op = vie.Operator(ctx, g)
    out[i] = [op.export_block(2, t) for t in range(len(g.sides))]
    op.close()
    ctx.close()


@pytest.mark.parametrize("nv", [1, 3, 4])
def test_grid_that_gives_up_runs_again(nv, monkeypatch):
    g = workloads.graded_array(2, nv, seed=1)   # three types
    from paper_2603_10586_gb300 import vie
    out, launches = [None, None], []
    for i, cycles in enumerate(("", "0")):
        monkeypatch.setenv("VIE_TEST_WAIT_CYCLES", cycles)
        n0 = vie.kernel_launches()
        _inverse(g, out, i)
        launches.append(vie.kernel_launches() - n0)
    assert launches[1] == launches[0] + len(g.sides)   # the second run of every type
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_two_contexts_at_the_same_time():
    g = workloads.single_cube(0.2, 7)
    out = [None] * 3
    _inverse(g, out, 0)
    th = [threading.Thread(target=_inverse, args=(g, out, i)) for i in (1, 2)]
    for t in th:
        t.start()
    for t in th:
        t.join()
    for o in out[1:]:
        assert o is not None and np.array_equal(o[0], out[0][0])
