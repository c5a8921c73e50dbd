"""The search for the OC multiplier (FP32 screening, then the exact bisection
over the few undecided elements) against the oracle's bisection over all
elements, and the inputs that it hands to the bisection over all elements.

Tolerance: the bisection stops at a relative width of 1e-9, so two runs of it
that round a volume differently differ by at most 2e-9 in lambda and 1e-9 in
x (x goes with lambda^(-1/2), x <= 1)."""
import numpy as np
import pytest

import synth
from gpu_common import n, t
from oracle import oc as ooc

pytestmark = pytest.mark.gpu
TOL = 2e-9


def _grid(dims):
    from paper_2201_12931_gb300 import Params, TopoGrid
    return TopoGrid(dims, Params(levels=1))


def _check(dims, x, dc, volfrac, move=0.2, passive=None):
    g = _grid(dims)
    want, change, _, _ = ooc.oc_update_unfiltered(x, dc, volfrac, move, passive=passive)
    xt = t(x)
    got = g.oc_update_unfiltered(move, volfrac, xt, t(dc), passive=None if passive is None else t(passive))
    assert np.abs(n(xt) - want).max() <= TOL
    assert abs(got - change) <= TOL
    g.close()


# one element, around a block of 256 and of 512, many blocks
@pytest.mark.parametrize("dims", [(1, 1, 1), (5, 17, 3), (16, 16, 1), (257, 1, 1), (8, 8, 8), (27, 19, 1), (64, 40, 41),
                                  (210, 90, 60)])
@pytest.mark.parametrize("volfrac", [0.05, 0.5])
def test_sizes(dims, volfrac):
    x = synth.uniform_field(dims, 81, 0.0, 1.0) if dims != (1, 1, 1) else np.array([volfrac])
    x *= volfrac / x.mean()
    _check(dims, x, -synth.uniform_field(dims, 82, 1e-6, 1.0) ** 3, volfrac, 0.1)


@pytest.mark.parametrize("scale", [1e-25, 1e-8, 1e6, 1e17])
def test_sensitivity_magnitudes(scale):
    """Multipliers from the low end of the bisection's range to its end at 1e9
    and, for 1e17, beyond it (everything at the upper bound)."""
    dims = (40, 20, 20)
    x = np.full(16000, 0.3)
    _check(dims, x, -scale * synth.uniform_field(dims, 83, 0.1, 1.0), 0.3)


def test_clamped_void_and_passive_elements():
    dims = (50, 21, 16)
    x = np.round(synth.uniform_field(dims, 84, 0.0, 1.0))            # 0 and 1: at the outer bounds
    dc = -synth.uniform_field(dims, 85, 0.0, 1.0) * x
    _check(dims, x, dc, 0.5)
    passive = (3 * synth.uniform_field(dims, 86)).astype(np.uint8)
    x = synth.uniform_field(dims, 87, 0.05, 0.6)
    x[passive == 1], x[passive == 2] = 1.0, 0.0
    _check(dims, x, -synth.uniform_field(dims, 88, 1e-3, 1.0), 0.3, 0.2, passive)


def test_many_elements_at_one_breakpoint():
    """Equal elements leave more undecided ones than the list holds: the
    multiplier at which all of them leave a bound is the root."""
    dims = (64, 40, 40)
    x = np.full(64 * 40 * 40, 0.3)
    dc = np.full(x.size, -1.0)
    x[::2] = 0.6
    dc[::2] = -0.2
    # the volume just where the even elements reach their lower bound
    _check(dims, x, dc, float(np.where(np.arange(x.size) % 2 == 0, 0.4, 0.3 * np.sqrt(5.0 * (0.4 / 0.6) ** 2)).mean()))


def test_values_outside_the_search():
    """A density above 1, a negative one, NaN and infinite sensitivities."""
    dims = (30, 10, 10)
    x = synth.uniform_field(dims, 89, 0.1, 0.9)
    dc = -synth.uniform_field(dims, 90, 1e-3, 1.0)
    dc[7] = np.nan
    want = dc.copy()
    want[7] = -1e-30                                                  # NaN counts as no sensitivity
    g = _grid(dims)
    xt = t(x)
    g.oc_update_unfiltered(0.2, 0.4, xt, t(dc))
    assert np.abs(n(xt) - ooc.oc_update_unfiltered(x, want, 0.4)[0]).max() <= TOL
    g.close()
    dc[7] = -np.inf
    _check(dims, x, dc, 0.4)
    x[11] = 1.1
    _check(dims, x, np.where(np.isinf(dc), -1.0, dc), 0.4)


def test_no_root_is_an_error():
    """All sensitivities zero and a target below the lower bounds: the
    bisection does not end, x stays as it was."""
    from paper_2201_12931_gb300 import TopoError
    dims = (12, 6, 6)
    g = _grid(dims)
    x = np.full(432, 0.5)
    xt = t(x)
    with pytest.raises(TopoError, match="bisection"):
        g.oc_update_unfiltered(0.1, 0.7, xt, t(np.zeros(432)))
    assert (n(xt) == x).all()
    # and the next call on the handle works
    dc = -synth.uniform_field(dims, 91, 0.1, 1.0)
    g.oc_update_unfiltered(0.2, 0.5, xt, t(dc))
    assert np.abs(n(xt) - ooc.oc_update_unfiltered(x, dc, 0.5)[0]).max() <= TOL
    g.close()


@pytest.mark.parametrize("dims,r", [((33, 18, 21), 1.5), ((60, 24, 24), 3.0)])
def test_filtered_update(dims, r):
    x = synth.uniform_field(dims, 92, 0.05, 0.6)
    dc = -synth.uniform_field(dims, 93, 1e-3, 1.0)
    g = _grid(dims)
    xt = t(x)
    got = g.oc_update(r, 0.1, 0.3, xt, t(dc))
    want, change, _, _ = ooc.oc_update(x, dc, dims, r, 0.3, 0.1)
    assert np.abs(n(xt) - want).max() <= TOL and abs(got - change) <= TOL
    g.close()
