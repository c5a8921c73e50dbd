"""The density filter neighbour by neighbour (thin, odd and small grids) and its
border to the march by symmetry classes: every number of neighbours along an axis,
rods and plates in each direction, grids that end inside a warp and inside a
block, and sizes on both sides of the choice, against the oracle's offset loops;
with and without scratch (the call without a handle), and with the properties that
the other filter tests ask of the march.

Tolerance: at most 905 positive-weight products added in different orders,
905 * 2^-53 = 1e-13 of the sum of their magnitudes; the random signs and the
usual cancellation of rounding leave 1e-14 of the largest result, the bar of the
other filter tests."""
import ctypes as C

import numpy as np
import pytest
import torch

import synth
from gpu_common import n, rel_max, t
from oracle import filter as oflt

pytestmark = pytest.mark.gpu

RADII = [0.8, 1.0, 1.2, 1.5, 2.0, 2.5, 3.0, 3.6, 4.2, 5.0, 5.5, 6.0]
THIN = [(1, 33, 40), (35, 1, 30), (31, 37, 1), (2, 3, 301), (2, 301, 3), (301, 2, 3), (4, 4, 65), (9, 11, 13), (33, 7, 8)]


def _check(dims, r):
    from paper_2201_12931_gb300 import Params, TopoGrid
    g = TopoGrid(dims, Params(levels=1))
    x = synth.uniform_field(dims, 171, -1.0, 1.0)
    rho = synth.uniform_field(dims, 172, 0.0, 1.0)
    dc = -synth.uniform_field(dims, 173, 1e-3, 1.0)
    H, HT = oflt.density_filter(x, dims, r), oflt.density_filter_T(x, dims, r)
    assert rel_max(n(g.filter(r, t(x))), H) <= 1e-14
    assert rel_max(n(g.filter(r, t(x), transpose=True)), HT) <= 1e-14
    want = oflt.density_filter(rho * dc, dims, r) / np.maximum(1e-3, rho)
    assert rel_max(n(g.sensitivity_filter(r, t(rho), t(dc))), want) <= 1e-14
    one = torch.ones(g.ne, dtype=torch.float64, device="cuda")
    assert (n(g.filter(r, one)) == 1.0).all()
    y = n(g.filter(r, t(np.round(synth.uniform_field(dims, 177, 0.0, 3.0)).clip(0.0, 1.0))))
    assert y.min() >= 0.0 and y.max() <= 1.0
    # H^T 1 through the update: the filtered volume of its result is the asked one
    # only if H^T 1 is right
    d = torch.full((g.ne,), 0.5, dtype=torch.float64, device="cuda")
    g.oc_update(r, 0.4, 0.45, d, t(dc))
    assert abs(oflt.density_filter(n(d), dims, r).mean() - 0.45) <= 1e-8
    for tr, ref in ((0, H), (1, HT)):
        out, xt = torch.empty(g.ne, dtype=torch.float64, device="cuda"), t(x)
        st = g.lib.topo_filter_noalloc(*dims, float(r), C.c_void_p(xt.data_ptr()), C.c_void_p(out.data_ptr()), tr,
                                       C.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert st == 0 and rel_max(n(out), ref) <= 1e-14
    g.close()


@pytest.mark.parametrize("r", RADII)
@pytest.mark.parametrize("dims", THIN)
def test_thin_and_small_grids(dims, r):
    _check(dims, r)


@pytest.mark.parametrize("r", [1.5, 2.5, 4.2])
@pytest.mark.parametrize("dims", [(20, 16, 12), (40, 21, 30), (75, 26, 33), (33, 120, 60), (64, 48, 40), (96, 64, 48)])
def test_both_sides_of_the_choice(dims, r):
    _check(dims, r)


@pytest.mark.parametrize("r", [1.0, 1.5, 2.3, 3.0])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_non_finite_values_reach_their_neighbourhood_only(r, value):
    from paper_2201_12931_gb300 import Params, TopoGrid
    dims = (3, 19, 20)
    g = TopoGrid(dims, Params(levels=1))
    x = synth.uniform_field(dims, 175, 0.1, 1.0)
    at = (1, 9, 10)
    x[at[0] + dims[0] * (at[1] + dims[1] * at[2])] = value
    k, j, i = np.meshgrid(*(np.arange(d) for d in dims[::-1]), indexing="ij")
    near = (np.sqrt((i - at[0]) ** 2 + (j - at[1]) ** 2 + (k - at[2]) ** 2) < r).ravel()
    for transpose in (False, True):
        y = n(g.filter(r, t(x), transpose=transpose))
        assert np.isfinite(y[~near]).all()
        assert np.isnan(y[near]).all() if np.isnan(value) else (y[near] == value).all()
    g.close()
