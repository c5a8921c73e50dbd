"""Calls on a stream that is being captured.  What a call keeps for later ones
(FP64 diagonals of a density, weights of a filter radius) has to have been
computed, not only recorded: a replayed sweep uses the density of the replay, a
direct call after the capture is right whether the graph ran or not, and a radius
whose weights are not there yet is refused, as the calls that wait for the
stream are.  Results are compared bit for bit with direct calls."""
import contextlib

import pytest
import torch

import synth
from gpu_common import cuda_device

pytestmark = pytest.mark.gpu

DIMS = (12, 6, 8)


def _setup(stream):
    from paper_2201_12931_gb300 import Params, TopoGrid
    with torch.cuda.stream(stream):
        g = TopoGrid(DIMS, Params(levels=2), stream=stream)
        pb = synth.mbb_half(DIMS)
        dev = cuda_device()
        rho = [torch.tensor(synth.uniform_field(DIMS, s, 0.1, 1.0), device=dev) for s in (5, 6)]
        g.set_density(rho[0])
        g.set_bc_loads(torch.tensor(pb.fixed, device=dev), torch.tensor(pb.f, device=dev))
        u, f = (torch.tensor(synth.uniform_field((3 * g.nn, 1, 1), s, -1.0, 1.0), device=dev) for s in (7, 8))
    stream.synchronize()
    return g, rho, u, f


@contextlib.contextmanager
def _refused(stream):
    """A capture in which the call has to fail; whether the capture itself
    survives the refused call is not what is tested."""
    from paper_2201_12931_gb300.api import TopoError
    try:
        with torch.cuda.graph(torch.cuda.CUDAGraph(), stream=stream):
            with pytest.raises(TopoError):
                yield
    except RuntimeError as e:
        if "captur" not in str(e).lower():
            raise
    torch.cuda.synchronize()


@pytest.mark.parametrize("fresh", [False, True])
def test_captured_sweep_follows_the_density(fresh):
    """fresh: the first sweep of a density is the captured one."""
    s = torch.cuda.Stream()
    g, rho, u, f = _setup(s)
    with torch.cuda.stream(s):
        g.jacobi_sweep(u, f)   # (workspace)
        if fresh:
            g.set_density(rho[0])
    s.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        out = g.jacobi_sweep(u, f)
    with torch.cuda.stream(s):
        g.set_density(rho[1])
        direct = [g.jacobi_sweep(u, f)] if fresh else []
        g.set_density(rho[1])
        graph.replay()
        first = out.clone()
        direct.append(g.jacobi_sweep(u, f))
        g.set_density(rho[0])
        graph.replay()
        second = out.clone()
        want = g.jacobi_sweep(u, f)
    s.synchronize()
    assert all(torch.equal(first, d) for d in direct)
    assert torch.equal(second, want) and not torch.equal(first, second)
    g.close()


def test_direct_sweep_after_a_capture_that_never_ran():
    s = torch.cuda.Stream()
    g, rho, u, f = _setup(s)
    with torch.cuda.stream(s):
        g.jacobi_sweep(u, f)
        g.set_density(rho[1])
        want = g.jacobi_sweep(u, f)
        g.set_density(rho[0])
        g.jacobi_sweep(u, f)
        g.set_density(rho[1])
    s.synchronize()
    with torch.cuda.graph(torch.cuda.CUDAGraph(), stream=s):
        g.jacobi_sweep(u, f)
    with torch.cuda.stream(s):
        got = g.jacobi_sweep(u, f)
    s.synchronize()
    assert torch.equal(got, want)
    g.close()


def test_new_filter_radius_is_refused():
    s = torch.cuda.Stream()
    g, rho, u, f = _setup(s)
    with torch.cuda.stream(s):
        want = g.filter(2.5, rho[0])
        old = g.filter(1.5, rho[0])
    s.synchronize()
    with _refused(s):
        g.filter(2.5, rho[0])
    with torch.cuda.stream(s):
        got = g.filter(2.5, rho[0])
        back = g.filter(1.5, rho[0])
    s.synchronize()
    assert torch.equal(got, want) and torch.equal(back, old)
    # a radius that is there can be captured
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        out = g.filter(1.5, rho[1])
    with torch.cuda.stream(s):
        graph.replay()
        want = g.filter(1.5, rho[1])
    s.synchronize()
    assert torch.equal(out, want)
    g.close()


def test_update_after_a_refused_capture():
    s = torch.cuda.Stream()
    g, rho, u, f = _setup(s)
    with torch.cuda.stream(s):
        dc = -torch.tensor(synth.uniform_field(DIMS, 9, 0.1, 1.0), device=cuda_device())
        want = rho[0].clone()
        g.oc_update(2.5, 0.2, 0.5, want, dc)
        g.oc_update(1.5, 0.2, 0.5, rho[0].clone(), dc)
        g.filter(2.5, rho[0])
        x = rho[0].clone()
    s.synchronize()
    with _refused(s):
        g.oc_update(2.5, 0.2, 0.5, x, dc)
    with torch.cuda.stream(s):
        x.copy_(rho[0])
        g.oc_update(2.5, 0.2, 0.5, x, dc)
    s.synchronize()
    assert torch.equal(x, want)
    g.close()
