"""The message of a failed coarsest-grid factorization names a degree of
freedom of the level, whatever order its rows are eliminated in: with void
corner elements (modulus exactly 0) the corner nodes have no stiffness, and the
smallest free DOF among them is the one reported, at every run alike."""
import re

import numpy as np
import pytest
import torch

import synth
from gpu_common import cuda_device

pytestmark = pytest.mark.gpu

DIMS = (12, 5, 4)   # eliminated from both ends: each void corner lies in a chain of its own


@pytest.mark.parametrize("graphs", [0, 1])
@pytest.mark.parametrize("corners", [("far",), ("near", "far"), ("near",)])
def test_message_names_the_dof(corners, graphs):
    from paper_2201_12931_gb300 import Params, TopoGrid, _lib
    nx, ny, nz = DIMS
    rho = np.ones((nz, ny, nx))
    nodes = []
    if "near" in corners:
        rho[0, 0, 0] = 0.0
        nodes.append(0)
    if "far" in corners:
        rho[-1, -1, -1] = 0.0
        nodes.append((nx + 1) * (ny + 1) * (nz + 1) - 1)
    pb = synth.mbb_half(DIMS)
    free = [3 * k + c for k in nodes for c in range(3) if not pb.fixed[3 * k + c]]
    g = TopoGrid(DIMS, Params(levels=1, Emin=0.0, graphs=graphs))
    g.set_density(torch.tensor(rho.ravel(), device=cuda_device()))
    g.set_bc_loads(torch.tensor(pb.fixed, device=cuda_device()), torch.tensor(pb.f, device=cuda_device()))
    for _ in range(3):
        _, res = g.solve(1e-8, 100, allow_breakdown=True)
        assert res.status == _lib.TOPO_BREAKDOWN
        row = re.search(r"row (\d+)", g.lib.topo_last_error(g._h).decode())
        assert row and int(row.group(1)) == min(free)
    g.close()
