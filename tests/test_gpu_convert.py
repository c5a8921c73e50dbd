"""FP64 <-> FP32 conversions of the step-level calls are the rounded values bit
for bit: with u = 0 the FP32 residual is fl32(f), widened.  Ties, the ends of
FP32's normal range, subnormals, zeros, infinities and NaN."""
import numpy as np
import pytest

import synth
from gpu_common import n, t

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(3, 4, 5), (60, 61, 62)])   # below and above the small-level limit
def test_residual_of_zero_rounds_the_load(dims):
    from paper_2201_12931_gb300 import Params, TopoGrid
    g = TopoGrid(dims, Params(levels=1, precision=1))
    g.set_density(t(np.full(g.ne, 0.5)))
    size = 3 * g.nn
    f = synth.uniform_field((size, 1, 1), 41, -1.0, 1.0) * 10.0 ** synth.uniform_field((size, 1, 1), 42, -45.0, 39.0)
    h = f[::3].astype(np.float32)
    f[::3] = 0.5 * (h.astype(np.float64) + np.nextafter(h, np.float32(np.inf)).astype(np.float64))   # ties
    big = float(np.finfo(np.float32).max)
    f[1:25] = [0.0, -0.0, np.inf, -np.inf, np.nan, big, -big, big * (1 + 2.0 ** -25), big * (1 + 2.0 ** -24), 1e300, -1e300,
               2.0 ** -126, 2.0 ** -127, -2.0 ** -149, 2.0 ** -150, 1.5 * 2.0 ** -150, 2.0 ** -126 * (1 - 2.0 ** -25),
               1e-300, 1.0, -1.0, 1 + 2.0 ** -24, 1 + 2.0 ** -23, 1 + 3 * 2.0 ** -24, -(1 + 3 * 2.0 ** -24)]
    with np.errstate(over="ignore"):
        want = f.astype(np.float32).astype(np.float64)
    got = n(g.residual(t(np.zeros(size)), t(f), 0, 1))
    nan = np.isnan(want)
    assert np.array_equal(nan, np.isnan(got))
    some = ~nan & (want != 0.0)
    assert (got[~nan & ~some] == 0.0).all()   # (f - 0: the sign of a zero is that of the difference)
    assert np.array_equal(got[some].view(np.uint64), want[some].view(np.uint64))
    g.close()
