"""The FP64 restriction on both sides of the number of blocks up to which a plane's
values are loaded before their masks (304), against the transpose of trilinear
interpolation formed axis by axis in numpy with both masks: 27 terms per node,
each rounded once or twice, 1e-14 of the largest entry."""
import numpy as np
import pytest

import synth
from gpu_common import n, rel_max, t

pytestmark = pytest.mark.gpu


def _axis(v, axis):
    """r_I = v_{2I-1} / 2 + v_{2I} + v_{2I+1} / 2 along one axis, zero outside."""
    v = np.moveaxis(v, axis, 0)
    r = v[::2].copy()
    r[1:] += 0.5 * v[1:-1:2]
    r[:-1] += 0.5 * v[1::2]
    return np.moveaxis(r, 0, axis)


@pytest.mark.parametrize("dims", [(16, 8, 8), (64, 64, 48), (64, 62, 76), (64, 62, 74), (88, 88, 88), (8, 8, 1000), (2000, 8, 8)])
def test_restriction(dims):
    from paper_2201_12931_gb300 import Params, TopoGrid
    g = TopoGrid(dims, Params(levels=2))
    pb = synth.mbb_half(dims)
    g.set_density(t(synth.uniform_field(dims, 181, 0.1, 1.0)))
    g.set_bc_loads(t(pb.fixed), t(pb.f))
    shape = (dims[2] + 1, dims[1] + 1, dims[0] + 1, 3)
    v = synth.uniform_field((3 * g.nn, 1, 1), 182, -1.0, 1.0)
    free = (pb.fixed == 0).reshape(shape)
    want = v.reshape(shape) * free
    for axis in range(3):
        want = _axis(want, axis)
    want = want * free[::2, ::2, ::2]
    assert rel_max(n(g.restrict(t(v))), want.ravel()) <= 1e-14
    g.close()
