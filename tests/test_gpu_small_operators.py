"""Operators of small levels: FP32 by bricks of 16 x 4 x 4 nodes, FP64 by
element columns of several layers with a node gather.  Grids whose node counts
lie on both sides of a brick, whose layers do not divide into columns, with
one element in a direction, and a V-cycle whose sweep takes the coarse
correction along; against the oracle's assembled operators.

Tolerances as in the operator parity tests: FP64 1e-12, FP32 1e-5 (a sweep
2e-5) of the largest entry -- about 20 terms per row, 1e-16 / 6e-8 each, with
the slack that cancellation between them needs; V-cycle FP32 1e-4."""
import pytest

import synth
from gpu_common import make_case, n, rel_max, t
from oracle import multigrid

pytestmark = pytest.mark.gpu

DIMS = [(1, 1, 1), (15, 3, 3), (16, 4, 4), (14, 2, 8), (17, 5, 1), (31, 7, 11), (33, 1, 9), (5, 23, 14), (47, 12, 7)]


@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 1e-5)])
@pytest.mark.parametrize("dims", DIMS)
def test_operator_sweep_residual(dims, precision, tol):
    g, pb, rho, H = make_case(dims, 1, seed=6)
    size = 3 * g.nn
    u = synth.uniform_field((size, 1, 1), 51, -1.0, 1.0)
    f = synth.uniform_field((size, 1, 1), 52, -1.0, 1.0)
    y = H[0].K @ u
    assert rel_max(n(g.apply_operator(t(u), 0, precision)), y) <= tol
    assert rel_max(n(g.residual(t(u), t(f), 0, precision)), f - y) <= tol
    assert rel_max(n(g.jacobi_sweep(t(u), t(f), 0, precision)), multigrid.jacobi(H[0], u, f, g.params.omega)) <= 2 * tol
    g.close()


@pytest.mark.parametrize("pre,post", [(2, 2), (1, 1), (2, 0), (0, 1), (3, 2)])
@pytest.mark.parametrize("dims,levels", [((12, 4, 8), 2), ((40, 8, 24), 4)])
def test_vcycle_sweep_counts(dims, levels, pre, post):
    """The coarse correction enters with the first post-sweep, or by itself
    when there is none."""
    g, pb, rho, H = make_case(dims, levels, seed=7, pre=pre, post=post)
    r = synth.uniform_field((3 * g.nn, 1, 1), 53, -1.0, 1.0) * (pb.fixed == 0)
    want = multigrid.vcycle(H, r, g.params.omega, pre, post)
    assert rel_max(n(g.vcycle(t(r), 0)), want) <= 1e-10
    assert rel_max(n(g.vcycle(t(r), 1)), want) <= 1e-4
    g.close()
