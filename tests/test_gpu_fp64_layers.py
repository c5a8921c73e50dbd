"""FP64 operators whose layers do not divide: element columns of several layers
with a shorter last one (levels of at most 2^20 elements), and z-march chunks
with a shorter last one, ragged tiles and more than 2^20 elements.  K u, residual
and sweep at every node against K0 applied element by element in numpy, 1e-12 of
the largest entry (about 200 roundings of 1e-16 a row; a sweep 2e-12); three CG
steps and a V-cycle against the same steps put together from the single
operators, 1e-10 (a few hundred roundings of the iterates, amplified by the step
lengths' own rounding)."""
import numpy as np
import pytest
import torch

import synth
from gpu_common import cuda_device, n, rel_max, t
from oracle import assemble, element
from oracle.grid import element_dofs

pytestmark = pytest.mark.gpu

COLUMNS = [(53, 46, 16), (47, 46, 27), (56, 37, 37), (59, 49, 35)]   # remainders 1 to 5 of 3 to 6 layers
MARCH = [(131, 97, 90), (152, 88, 80), (40, 203, 131)]               # above 2^20 elements


def _layers_per_column(dims, sms):
    """The plan's choice: time of the fullest warp scheduler in both kernels."""
    nx, ny, nz = dims
    nodes, units, best = (nx + 1) * (ny + 1) * (nz + 1), 4 * sms, None
    for cz in range(1, min(8, nz) + 1):
        warps = -(-nx * ny * -(-nz // cz) // 32)
        cost = (-(-warps // units) * (48.0 * (cz + 1) + 80.0 * cz + 12.0 * (cz - 1))
                + -(-nodes // (32 * units)) * (15.0 + 12.0 / cz))
        if best is None or cost < best[0]:
            best = (cost, cz)
    return best[1]


def _grid(dims, levels):
    from paper_2201_12931_gb300 import Params, TopoGrid
    g = TopoGrid(dims, Params(levels=levels, precision=0))
    pb = synth.mbb_half(dims)
    rho = synth.uniform_field(dims, 71, 1e-2, 1.0)
    g.set_density(t(rho))
    g.set_bc_loads(t(pb.fixed), t(pb.f))
    return g, pb, rho


@pytest.mark.parametrize("dims", COLUMNS + MARCH)
def test_operator_residual_sweep(dims):
    g, pb, rho = _grid(dims, 1)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if dims in MARCH:
        assert g.ne > 2 ** 20
    elif sms == 152:
        cz = _layers_per_column(dims, sms)
        assert cz >= 3 and dims[2] % cz != 0
    u, f = (synth.uniform_field((3 * g.nn, 1, 1), s, -1.0, 1.0) for s in (72, 73))
    fixed = pb.fixed.astype(bool)
    K0, E, edof = element.element_stiffness(0.3), assemble.simp_modulus(rho), element_dofs(dims)
    loc = np.where(fixed, 0.0, u)[edof] @ K0
    loc *= E[:, None]
    y = np.bincount(edof.ravel(), loc.ravel(), minlength=u.size)
    y[fixed] = u[fixed]
    D = np.bincount(edof.ravel(), np.repeat(E, 24) * K0[0, 0], minlength=u.size)   # (the diagonal of K0 is uniform)
    D[fixed] = 1.0
    assert rel_max(n(g.apply_operator(t(u), 0, 0)), y) <= 1e-12
    assert rel_max(n(g.residual(t(u), t(f), 0, 0)), f - y) <= 1e-12
    assert rel_max(n(g.jacobi_sweep(t(u), t(f), 0, 0)), u + g.params.omega * (f - y) / D) <= 2e-12
    g.close()


@pytest.mark.parametrize("dims,levels", [((68, 36, 32), 3), ((152, 88, 80), 4)])
def test_cg_steps_and_vcycle(dims, levels):
    from paper_2201_12931_gb300 import Params, TopoGrid
    g, pb, rho = _grid(dims, levels)
    f = t(np.where(pb.fixed != 0, 0.0, pb.f))
    # V-cycle: the coarse correction from a handle whose finest level is the next coarser one
    half = tuple(d // 2 for d in dims)
    h = TopoGrid(half, Params(levels=levels - 1, precision=0, E0=2.0, Emin=2e-9))
    nodes = pb.fixed.reshape(dims[2] + 1, dims[1] + 1, dims[0] + 1, 3)[::2, ::2, ::2]
    h.set_density(g.level_density(1))
    h.set_bc_loads(t(nodes.ravel()), torch.zeros(3 * h.nn, dtype=torch.float64, device=cuda_device()))
    r = t(synth.uniform_field((3 * g.nn, 1, 1), 74, -1.0, 1.0) * (pb.fixed == 0))
    u = torch.zeros_like(r)
    for _ in range(2):
        u = g.jacobi_sweep(u, r)
    u = g.prolong_add(h.vcycle(g.restrict(g.residual(u, r))), u)
    for _ in range(2):
        u = g.jacobi_sweep(u, r)
    assert rel_max(n(g.vcycle(r)), n(u)) <= 1e-10
    # three steps of CG
    x, r = torch.zeros_like(f), f.clone()
    z = g.vcycle(r)
    p, rz = z, torch.dot(r, z)
    for k in range(3):
        q = g.apply_operator(p)
        alpha = rz / torch.dot(p, q)
        x, r = x + alpha * p, r - alpha * q
        z = g.vcycle(r)
        old, rz = rz, torch.dot(r, z)
        p = z + rz / old * p
    got = torch.empty_like(x)
    _, res = g.solve(1e-30, 3, out=got)
    assert res.iters == 3
    assert rel_max(n(got), n(x)) <= 1e-10
    g.close()
    h.close()
