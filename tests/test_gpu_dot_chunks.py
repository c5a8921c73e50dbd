"""Norms formed inside the z-march do not lose more the longer a chunk of planes
is.  A grid whose 152 tiles of nodes fill the GPU marches over all of its 97
planes in one chunk; with moduli of 1e-30 the residual is the load, and the load
is 1 on the first plane and 2^-13 on the others, so that an FP32 sum of squares
carried over the whole column (its ulp is 2^-22 after the first plane) drops
every later 2^-26: 96 planes are 1.4e-6 of the square, 7.2e-7 of the norm.  Sums
of at most eight planes drop those of the first group only, 5.2e-8 of the
norm."""
import numpy as np
import pytest
import torch

import synth
from gpu_common import cuda_device

pytestmark = pytest.mark.gpu


def test_norm_of_a_long_column():
    from paper_2201_12931_gb300 import Params, TopoGrid, _lib
    dims = (240, 128, 96)
    dev = cuda_device()
    g = TopoGrid(dims, Params(levels=5, precision=1, Emin=1e-30))
    pb = synth.cantilever(dims)
    f = torch.full((dims[2] + 1, 3 * (dims[0] + 1) * (dims[1] + 1)), 2.0 ** -13, dtype=torch.float64, device=dev)
    f[0] = 1.0
    f = f.ravel().contiguous()
    g.set_bc_loads(torch.tensor(pb.fixed, device=dev), f)
    g.set_density(torch.ones(g.ne, dtype=torch.float64, device=dev))
    _, res = g.solve(1e-6, 1)                 # any solution that is not zero
    assert res.status == _lib.TOPO_MAXITER
    g.set_density(torch.zeros(g.ne, dtype=torch.float64, device=dev))
    _, res = g.solve(10.0, 1)                 # no iteration: the norm of f - K x alone
    assert res.iters == 0
    assert abs(res.relres - 1.0) <= 1e-7
    g.close()
