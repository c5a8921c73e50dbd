"""Factor and inverse of the coarsest grid by blocks of 32: one level, so that
the V-cycle is the direct solve, at orders below a block's multiple, on it (96,
288) and just past it (225), eliminated from both ends (225 and more) and not,
with moduli over nine orders of magnitude.  The tolerance is the order times the
condition number of the matrix scaled to a unit diagonal times 2^-53, from the
matrix itself."""
import numpy as np
import pytest

import synth
from gpu_common import make_case, n, rel_max, t
from oracle import multigrid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(1, 3, 3), (4, 4, 2), (2, 2, 2), (3, 3, 5), (1, 2, 1), (6, 1, 2), (12, 5, 4), (40, 1, 1)])
@pytest.mark.parametrize("lo", [1e-3, 0.3])
def test_direct_solve(dims, lo):
    g, pb, rho, H = make_case(dims, 1, seed=91, lo=lo)
    r = synth.uniform_field((H[0].K.shape[0], 1, 1), 92, -1, 1)
    r[pb.fixed.astype(bool)] = 0.0
    z = n(g.vcycle(t(r), precision=0))
    K = H[0].K.toarray()
    d = 1.0 / np.sqrt(K.diagonal())
    tol = K.shape[0] * np.linalg.cond(d[:, None] * K * d) * 2.0 ** -53
    assert rel_max(z, multigrid.vcycle(H, r, g.params.omega, g.params.pre, g.params.post)) <= tol
    g.close()
