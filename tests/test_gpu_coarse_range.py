"""The FP32 coarsest solve at the ends of FP32's exponent range: its triangular
products give what FP64 sums of the same terms give, also where single terms lie
beyond FP32's largest value and cancel, or far below 1.  One level, so that the
V-cycle is the solve.  The solution is a displacement of alternating sign in a
slender beam: in the product with W^T single terms are 6 to 20 times the result
(in any order of elimination) and the terms of a row add up to at most 512 times
it.  Scaled by a power of two every operation scales exactly, up to a last bit of
the intermediate vector (2^-23 of each term), so the solution does too within
512 * 2^-23 of its largest entry."""
import numpy as np
import pytest

import synth
from gpu_common import make_case, n, t

pytestmark = pytest.mark.gpu

TOL = 512 * 2.0 ** -23


@pytest.mark.parametrize("top", [127, 126, 122, 60, 0, -60, -80])
def test_scaled_direct_solve(top):
    """top: the binary exponent of the largest entry of the solution."""
    E0 = 2.0 ** -20
    g, pb, rho, H = make_case((24, 1, 1), 1, seed=91, lo=0.3, E0=E0, Emin=E0 * 1e-9)
    u = np.sign(synth.uniform_field((3 * g.nn, 1, 1), 93, -1.0, 1.0)) * (pb.fixed == 0)
    r = (H[0].K @ u).astype(np.float32).astype(np.float64)
    base = n(g.vcycle(t(r), precision=1))
    largest = np.abs(base).max()
    shift = top - int(np.floor(np.log2(largest)))
    assert np.abs(r).max() * 2.0 ** shift < 2.0 ** 120
    got = n(g.vcycle(t(r * 2.0 ** shift), precision=1)) * 2.0 ** -shift
    assert np.isfinite(got).all()
    assert np.abs(got - base).max() <= TOL * largest
    g.close()
