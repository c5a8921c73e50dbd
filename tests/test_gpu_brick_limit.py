"""FP32 operators on both sides of the node count where bricks give way to the
z-march (80000), against K0 applied element by element in numpy at every node:
1e-5 of the largest entry, a sweep 2e-5, and a V-cycle against the FP64 one 1e-4,
the tolerances of the operator parity tests."""
import numpy as np
import pytest

import synth
from gpu_common import n, rel_max, t
from oracle import assemble, element
from oracle.grid import element_dofs

pytestmark = pytest.mark.gpu


def _grid(dims, levels):
    from paper_2201_12931_gb300 import Params, TopoGrid
    g = TopoGrid(dims, Params(levels=levels, precision=1))
    pb = synth.mbb_half(dims)
    rho = synth.uniform_field(dims, 75, 1e-2, 1.0)
    g.set_density(t(rho))
    g.set_bc_loads(t(pb.fixed), t(pb.f))
    return g, pb, rho


@pytest.mark.parametrize("dims,brick", [((42, 43, 41), True), ((43, 43, 41), False), ((99, 398, 1), True), ((15, 61, 80), False)])
def test_operator_residual_sweep(dims, brick):
    g, pb, rho = _grid(dims, 1)
    assert (g.nn <= 80000) == brick and 79000 < g.nn < 82000
    u, f = (synth.uniform_field((3 * g.nn, 1, 1), s, -1.0, 1.0).astype(np.float32).astype(np.float64) for s in (76, 77))
    fixed = pb.fixed.astype(bool)
    K0, E, edof = element.element_stiffness(0.3), assemble.simp_modulus(rho), element_dofs(dims)
    loc = (np.where(fixed, 0.0, u)[edof] @ K0) * E[:, None]
    y = np.bincount(edof.ravel(), loc.ravel(), minlength=u.size)
    y[fixed] = u[fixed]
    D = np.bincount(edof.ravel(), np.repeat(E, 24) * K0[0, 0], minlength=u.size)
    D[fixed] = 1.0
    assert rel_max(n(g.apply_operator(t(u), 0, 1)), y) <= 1e-5
    assert rel_max(n(g.residual(t(u), t(f), 0, 1)), f - y) <= 1e-5
    assert rel_max(n(g.jacobi_sweep(t(u), t(f), 0, 1)), u + g.params.omega * (f - y) / D) <= 2e-5
    g.close()


@pytest.mark.parametrize("dims", [(48, 40, 36), (48, 44, 36)])
def test_vcycle(dims):
    g, pb, _ = _grid(dims, 3)
    r = t(synth.uniform_field((3 * g.nn, 1, 1), 78, -1.0, 1.0) * (pb.fixed == 0))
    assert rel_max(n(g.vcycle(r, 1)), n(g.vcycle(r, 0))) <= 1e-4
    g.close()
