"""Device memory that a call takes on first use is what the call needs: the
double-FP32 product of a mixed handle allocates the FP64 vectors of the levels
(as every FP64 step call does) but not the element scratch of the FP64
operators, which the first of those takes."""
import pytest
import torch

import synth
from gpu_common import cuda_device

pytestmark = pytest.mark.gpu


def test_double_fp32_product_takes_no_element_scratch():
    from paper_2201_12931_gb300 import Params, TopoGrid, TOPO_DF32, TOPO_FP64
    dims = (96, 96, 96)
    dev = cuda_device()
    g = TopoGrid(dims, Params(levels=3, precision=1))
    pb = synth.cantilever(dims)
    g.set_density(torch.ones(g.ne, dtype=torch.float64, device=dev))
    g.set_bc_loads(torch.tensor(pb.fixed, device=dev), torch.tensor(pb.f, device=dev))
    u = torch.ones(3 * g.nn, dtype=torch.float64, device=dev)
    y = torch.empty_like(u)

    def growth(call):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        call()
        torch.cuda.synchronize()
        return before - torch.cuda.mem_get_info()[0]

    def apply(precision):
        g._check(g.lib.topo_apply_operator(g._h, 0, precision, u.data_ptr(), y.data_ptr()))

    # three vectors per level, nine more on the finest; 2 MiB granules
    nodes = [g.level_nodes(l) for l in range(3)]
    vectors = 8 * 3 * (3 * sum(nodes) + 9 * nodes[0]) + 18 * (2 << 20)
    assert growth(lambda: apply(TOPO_DF32)) <= vectors
    assert growth(lambda: apply(TOPO_DF32)) == 0
    assert growth(lambda: apply(TOPO_FP64)) >= 8 * 12 * g.ne   # at least one face of 12 values per element
    assert growth(lambda: apply(TOPO_FP64)) == 0
    g.close()
