"""Products whose convolution passes are chained: queued back to back without a wait, each with
its own input, they give what each gives alone (bit for bit: the passes have no atomics), for one
column and several and for lengths from 16 to past the chained range; captured into a graph (no
chaining there) they give the same.  Against the FP64 oracle: the framework's 1e-6."""
import numpy as np
import pytest
import torch

import oracle
import paper_2501_04684_gb300 as ie
import workloads as W
from gpu_util import dev, empty, host, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("extent,nrhs", [((4, 4, 4), 1), ((4, 4, 4), 3), ((5, 9, 13), 2), ((3, 3, 33), 1)])
def test_queued_products(extent, nrhs):
    g = W.rng(880 + extent[2] + nrhs)
    ijk = np.stack(np.meshgrid(*[np.arange(e) for e in extent], indexing="ij"), -1).reshape(-1, 3).astype(np.int32)
    ijk = ijk[g.permutation(len(ijk))]
    nb = np.full(len(ijk), 8, dtype=np.int32)
    p = W.Problem(name="chain", G=max(extent), box_ijk=ijk, nb=nb, P=W.random_P(g, nb), alpha=4.0e6)
    cs = [W.coefficients(p, nrhs, 881 + i) for i in range(6)]
    with ie.Plan(ie.problem_from(p, ie.precmask(ie.IE_PREC_FP32), nrhs)) as plan:
        xs = [dev(c) for c in cs]
        alone = []
        for x in xs:
            y = empty((nrhs, p.n))
            ie.ie_matvec(plan.handle, ie.IE_FULL, ie.IE_PREC_FP32, x, y, nrhs)
            torch.cuda.synchronize()
            alone.append(host(y))
        assert rel_l2(alone[0], oracle.operator(p, cs[0], "full")) <= 1e-6
        ys = [empty((nrhs, p.n)) for _ in xs]
        for _ in range(5):
            for x, y in zip(xs, ys):
                ie.ie_matvec(plan.handle, ie.IE_FULL, ie.IE_PREC_FP32, x, y, nrhs)
        torch.cuda.synchronize()
        for y, a in zip(ys, alone):
            assert np.array_equal(host(y), a)
        y = empty((nrhs, p.n))
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            ie.ie_matvec(plan.handle, ie.IE_FULL, ie.IE_PREC_FP32, xs[1], y, nrhs)
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(host(y), alone[1])
