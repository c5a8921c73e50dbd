"""Operators of levels above the limits of the small-level kernels (200000
nodes in FP32), with ragged last tiles and chunks of every length modulo the
groups of four planes that the z-march takes.  The FP64 operators are checked
against the oracle's rows at sampled nodes (1e-12 of the largest entry), the
FP32 ones against them at every node: 1e-5, a sweep 2e-5, the V-cycle 1e-4,
the tolerances of the parity tests.  Inputs are not zero at fixed DOFs: the
step-level calls keep the identity rows there."""
import numpy as np
import pytest
import torch

import synth
from gpu_common import cuda_device, n, rel_max
from oracle import assemble, element

pytestmark = pytest.mark.gpu

DIMS = [(67, 59, 53), (63, 64, 52), (62, 55, 60), (201, 31, 40), (31, 70, 95), (700, 17, 17), (8, 9, 2400), (64, 60, 56)]


def _grid(dims, levels, problem="mbb"):
    from paper_2201_12931_gb300 import Params, TopoGrid
    g = TopoGrid(dims, Params(levels=levels, precision=1))
    pb = synth.mbb_half(dims) if problem == "mbb" else synth.cantilever(dims)
    rho = synth.uniform_field(dims, 61, 1e-3, 1.0)
    g.set_density(torch.tensor(rho, device=cuda_device()))
    g.set_bc_loads(torch.tensor(pb.fixed, device=cuda_device()), torch.tensor(pb.f, device=cuda_device()))
    return g, pb, rho


def _vector(g, seed):
    v = synth.uniform_field((3 * g.nn, 1, 1), seed, -1.0, 1.0).astype(np.float32).astype(np.float64)
    return v, torch.tensor(v, device=cuda_device())


@pytest.mark.parametrize("dims", DIMS)
def test_operator_sweep_residual(dims):
    g, pb, rho = _grid(dims, 1)
    assert g.nn > 200000
    u, ut = _vector(g, 62)
    f, ft = _vector(g, 63)
    y64 = n(g.apply_operator(ut, 0, 0))
    nodes = synth.sample_without_replacement(64, g.nn, 60)
    E = assemble.simp_modulus(rho, 1.0, 1e-9, 3.0)
    ref = assemble.operator_rows(dims, nodes, lambda e: E[e], lambda d: u[d], element.element_stiffness(0.3),
                                 lambda d: pb.fixed[d])
    idx = (3 * np.asarray(nodes)[:, None] + np.arange(3)).ravel()
    assert np.abs(y64[idx].reshape(-1, 3) - ref).max() <= 1e-12 * np.abs(y64).max()
    assert rel_max(n(g.apply_operator(ut, 0, 1)), y64) <= 1e-5
    assert rel_max(n(g.residual(ut, ft, 0, 1)), f - y64) <= 1e-5
    assert rel_max(n(g.jacobi_sweep(ut, ft, 0, 1)), n(g.jacobi_sweep(ut, ft, 0, 0))) <= 2e-5
    g.close()


@pytest.mark.parametrize("pre,post", [(2, 2), (3, 1), (1, 0)])
def test_vcycle(pre, post):
    from paper_2201_12931_gb300 import Params, TopoGrid
    dims = (80, 48, 64)
    out = []
    for precision in (0, 1):
        g = TopoGrid(dims, Params(levels=5, precision=precision, pre=pre, post=post))
        pb = synth.mbb_half(dims)
        g.set_density(torch.tensor(synth.uniform_field(dims, 65, 1e-3, 1.0), device=cuda_device()))
        g.set_bc_loads(torch.tensor(pb.fixed, device=cuda_device()), torch.tensor(pb.f, device=cuda_device()))
        _, r = _vector(g, 66)
        out.append(n(g.vcycle(r, precision)))
        g.close()
    assert rel_max(out[1], out[0]) <= 1e-4


def test_solve_against_fp64():
    from paper_2201_12931_gb300 import Params, TopoGrid
    dims, u = (104, 56, 48), []
    for precision in (0, 1):
        g = TopoGrid(dims, Params(levels=4, precision=precision))
        pb = synth.cantilever(dims)
        g.set_density(torch.tensor(synth.uniform_field(dims, 67, 0.05, 1.0), device=cuda_device()))
        g.set_bc_loads(torch.tensor(pb.fixed, device=cuda_device()), torch.tensor(pb.f, device=cuda_device()))
        v = torch.empty(3 * g.nn, dtype=torch.float64, device=cuda_device())
        _, res = g.solve(1e-9, 2000, out=v)
        assert res.status == 0
        u.append(n(v))
        assert (u[-1][pb.fixed.astype(bool)] == 0.0).all()
        g.close()
    # both residuals are below 1e-9 of the load; the displacement amplifies a
    # residual by at most the spread of the smooth modes, a few hundred here
    assert np.linalg.norm(u[1] - u[0]) <= 1e-6 * np.linalg.norm(u[0])
