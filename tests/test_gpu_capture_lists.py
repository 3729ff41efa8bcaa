"""Products captured into a graph after other products of the same plan have run: what the
first call of a kind prepares on the device does not depend on which call came before."""
import numpy as np
import pytest
import torch

import oracle
import paper_2501_04684_gb300 as ie
import workloads as W
from gpu_util import dev, empty, host, rel_l2

pytestmark = pytest.mark.gpu
BOUND = {ie.IE_PREC_FP32: 1e-6, ie.IE_PREC_FP16X3: 2e-6, ie.IE_PREC_FP16X1: 2e-3}


@pytest.mark.parametrize("symmetry", [0, 1])
@pytest.mark.parametrize("warm,captured", [((ie.IE_FULL, ie.IE_PREC_FP16X3), (ie.IE_FAR, ie.IE_PREC_FP16X3)),
                                           ((ie.IE_FULL, ie.IE_PREC_FP16X3), (ie.IE_FAR, ie.IE_PREC_FP16X1)),
                                           ((ie.IE_FULL, ie.IE_PREC_FP16X3), (ie.IE_FULL, ie.IE_PREC_FP16X1)),
                                           ((ie.IE_FULL, ie.IE_PREC_FP32), (ie.IE_FAR, ie.IE_PREC_FP32))])
def test_capture_after_another_product(warm, captured, symmetry):
    g = W.rng(990)
    ijk = W.full_grid(5)
    nb = np.full(len(ijk), 8, np.int32)
    p = W.Problem(name="capture", G=5, box_ijk=ijk, nb=nb, P=W.random_P(g, nb), alpha=4e6)
    c = W.coefficients(p, 2, 991)
    with ie.Plan(ie.problem_from(p, ie.precmask(*BOUND), 2, symmetry=symmetry)) as plan:
        assert ie.ie_plan_far_bytes(plan.handle, ie.IE_FAR, ie.IE_PREC_FP16X3, 2) > 0
        x, y = dev(c), empty((2, p.n))
        ie.ie_matvec(plan.handle, *warm, x, y, 2)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            ie.ie_matvec(plan.handle, *captured, x, y, 2)
        y.zero_()
        graph.replay()
        ref = oracle.far_matvec(p, c) if captured[0] == ie.IE_FAR else oracle.operator(p, c, "full")
        assert rel_l2(host(y), ref) <= BOUND[captured[1]]
        eager = empty((2, p.n))
        ie.ie_matvec(plan.handle, *captured, x, eager, 2)
        assert rel_l2(host(eager), ref) <= BOUND[captured[1]]
