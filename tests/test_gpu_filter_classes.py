"""The density filter summed by symmetry classes: every offset class, cut
neighbourhoods on grids thinner than the radius, tile edges, the sensitivity
filter and non-finite values, against the oracle's offset loops.

Tolerance: both sides add at most 905 positive-weight products in different
orders, at most 905 * 2^-53 = 1e-13 of the sum of their magnitudes; the
random signs and the usual cancellation of rounding leave 1e-14 of the
largest result, the bar of the other filter tests."""
import numpy as np
import pytest

import synth
from gpu_common import n, rel_max, t
from oracle import filter as oflt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,r", [
    ((1, 1, 7), 3.0), ((3, 2, 5), 6.0), ((11, 10, 1), 5.5), ((2, 40, 3), 2.5),   # thinner than the radius
    ((16, 8, 9), 0.7), ((17, 9, 5), 1.0), ((33, 5, 4), 1.01),                    # no neighbours, tile edges
    ((31, 4, 12), 1.5), ((65, 13, 7), 2.0), ((48, 17, 11), 2.3),
    ((34, 12, 20), 3.0), ((30, 21, 16), 3.7), ((19, 23, 15), 4.6), ((26, 14, 13), 6.0)])
def test_filter_and_transpose(dims, r):
    from paper_2201_12931_gb300 import Params, TopoGrid
    g = TopoGrid(dims, Params(levels=1))
    x = synth.uniform_field(dims, 71, -1.0, 1.0)
    rho = synth.uniform_field(dims, 72, 0.0, 1.0)
    dc = -synth.uniform_field(dims, 73, 1e-3, 1.0)
    assert rel_max(n(g.filter(r, t(x))), oflt.density_filter(x, dims, r)) <= 1e-14
    assert rel_max(n(g.filter(r, t(x), transpose=True)), oflt.density_filter_T(x, dims, r)) <= 1e-14
    want = oflt.density_filter(rho * dc, dims, r) / np.maximum(1e-3, rho)
    assert rel_max(n(g.sensitivity_filter(r, t(rho), t(dc))), want) <= 1e-14
    g.close()


def test_long_thin_grid():
    """More tiles along y and chunks along z than a grid dimension of 65535 holds."""
    from paper_2201_12931_gb300 import Params, TopoGrid
    for dims in ((1, 300000, 1), (1, 1, 300000), (300000, 1, 1)):
        g = TopoGrid(dims, Params(levels=1))
        x = synth.uniform_field(dims, 74)
        assert rel_max(n(g.filter(1.5, t(x))), (lambda v, w: v / w)(
            np.convolve(x, [0.5, 1.5, 0.5], "same"), np.convolve(np.ones_like(x), [0.5, 1.5, 0.5], "same"))) <= 1e-14
        g.close()


@pytest.mark.parametrize("r", [1.5, 2.3, 3.0])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_non_finite_values_reach_their_neighbourhood_only(r, value):
    from paper_2201_12931_gb300 import Params, TopoGrid
    dims = (37, 9, 10)
    g = TopoGrid(dims, Params(levels=1))
    x = synth.uniform_field(dims, 75, 0.1, 1.0)
    at = (18, 4, 5)
    x[at[0] + dims[0] * (at[1] + dims[1] * at[2])] = value
    k, j, i = np.meshgrid(*(np.arange(d) for d in dims[::-1]), indexing="ij")
    near = (np.sqrt((i - at[0]) ** 2 + (j - at[1]) ** 2 + (k - at[2]) ** 2) < r).ravel()
    for transpose in (False, True):
        y = n(g.filter(r, t(x), transpose=transpose))
        assert np.isfinite(y[~near]).all()
        assert np.isnan(y[near]).all() if np.isnan(value) else (y[near] == value).all()
    g.close()


def test_extreme_magnitudes():
    """Values at the ends of the exponent range keep the plain division."""
    from paper_2201_12931_gb300 import Params, TopoGrid
    dims = (20, 6, 6)
    g = TopoGrid(dims, Params(levels=1))
    for scale in (0.0, 1e-300, 1e300):
        x = scale * synth.uniform_field(dims, 76, 0.1, 1.0)
        got, want = n(g.filter(2.5, t(x))), oflt.density_filter(x, dims, 2.5)
        assert np.abs(got - want).max() <= 1e-14 * scale
    g.close()


@pytest.mark.parametrize("dims,r", [((40, 11, 9), 1.5), ((35, 13, 17), 3.0), ((4, 9, 21), 5.3)])
def test_unit_interval_is_kept(dims, r):
    """H maps [0, 1] into [0, 1] and ones to ones, in every bit: set_density
    refuses a density above 1 by one rounding."""
    from paper_2201_12931_gb300 import Params, TopoGrid
    g = TopoGrid(dims, Params(levels=1))
    one = np.ones(dims[0] * dims[1] * dims[2])
    assert (n(g.filter(r, t(one))) == 1.0).all()
    x = np.round(synth.uniform_field(dims, 77, 0.0, 3.0)).clip(0.0, 1.0)   # mostly plateaus of 1
    y = n(g.filter(r, t(x)))
    assert y.min() >= 0.0 and y.max() <= 1.0
    g.close()
