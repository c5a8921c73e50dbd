"""The root and the quotient of the OC candidate, to the last bits.  With move
limits that bind nowhere, x_new = x (-dc / dv)^(1/2) lambda^(-1/2) for one lambda,
so x_new / (x (-dc / dv)^(1/2)) is the same number for all elements.  Roundings:
the root 2^-52, the two products 2^-53 each, hence a spread of 2^-50 between the
largest and the smallest of these ratios; with a quotient of 2^-52 below the
root, half of that more each way, 2^-50 + 2^-52.  The scale of dc goes from the
floor of 1e-30 over both ends of the range that the short form of the root takes
(2^-101, 2^60)."""
import numpy as np
import pytest
import torch

import synth
from gpu_common import cuda_device, n, t

pytestmark = pytest.mark.gpu

DIMS = (20, 10, 8)   # small enough that every element's weight sum is its own
LD = np.longdouble


def _case(k, seed):
    """x of a size at which the multiplier stays below 1e9, dc = -2^k (1 .. 4)."""
    from paper_2201_12931_gb300 import Params, TopoGrid
    assert np.finfo(LD).eps < 2.0 ** -60
    g = TopoGrid(DIMS, Params(levels=1))
    x = (0.5 + 0.5 * synth.uniform_field(DIMS, seed, 0.0, 1.0)) * 2.0 ** -max(0, k // 2 - 8)
    dc = -(2.0 ** k) * (1.0 + 3.0 * synth.uniform_field(DIMS, seed + 1, 0.0, 1.0))
    return g, x, dc


def _spread(x_new, x, B):
    q = x_new.astype(LD) / (x.astype(LD) * np.sqrt(B.astype(LD)))
    return float(q.max() / q.min() - 1)


@pytest.mark.parametrize("k", [-110, -100, -99, -61, -20, -1, 0, 1, 30, 57, 58, 59, 60, 61])
def test_root(k):
    g, x, dc = _case(k, 81)
    xt = t(x)
    g.oc_update_unfiltered(1.0, 0.25, xt, t(dc))
    new = n(xt)
    assert new.max() < 1.0 and new.min() > 0.0 and abs(new.mean() - 0.25) < 1e-8
    assert _spread(new, x, np.maximum(-dc, 1e-30)) <= 2.0 ** -50
    g.close()


@pytest.mark.parametrize("r", [1.5, 2.5])
@pytest.mark.parametrize("k", [-98, -40, 0, 29, 57, 58, 61])
def test_root_of_a_quotient(k, r):
    g, x, dc = _case(k, 83)
    xt = t(x)
    dct = n(g.filter(r, t(dc), transpose=True))
    dv = n(g.filter(r, torch.ones(g.ne, dtype=torch.float64, device=cuda_device()), transpose=True))
    g.oc_update(r, 1.0, 0.25, xt, t(dc))
    new = n(xt)
    assert new.max() < 1.0 and new.min() > 0.0
    assert _spread(new, x, np.maximum(-dct, 1e-30).astype(LD) / dv.astype(LD)) <= 2.0 ** -50 + 2.0 ** -52
    g.close()
