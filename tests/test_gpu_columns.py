"""The products that share a read of P and of the near blocks between right-hand sides, at the
edges of their tiles: one to five columns (a full group of four, its remainders, one more) and
boxes of 1, 31, 32, 33, 64, 65 and 192 basis functions.  Bound: the framework's 1e-6 relative
L2 against the FP64 oracle."""
import numpy as np
import pytest

import oracle
import paper_2501_04684_gb300 as ie
import workloads as W
from gpu_util import dev, empty, host, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("largest", [32, 64, 192])
@pytest.mark.parametrize("nrhs", [1, 2, 3, 4, 5])
def test_mapping_and_near_products(largest, nrhs):
    g = W.rng(770 + nrhs + largest)
    ijk = W.full_grid(2)[g.permutation(8)].astype(np.int32)
    sizes = np.array([1, 31, 32, 17, 33, 64, 65, 192], dtype=np.int32)
    nb = np.minimum(sizes, largest)[g.permutation(8)]
    nb[0] = largest
    p = W.Problem(name="cols", G=2, box_ijk=ijk, nb=nb, P=W.random_P(g, nb), alpha=4.0e6)
    c = W.coefficients(p, nrhs, 771)
    X = oracle.aggregate(p, c)
    with ie.Plan(ie.problem_from(p, ie.precmask(ie.IE_PREC_FP32), nrhs)) as plan:
        Xg, r, y = empty((nrhs, p.n_boxes, W.NU)), empty((nrhs, p.n)), empty((nrhs, p.n))
        ie.ie_aggregate(plan.handle, dev(c), Xg, nrhs)
        assert rel_l2(host(Xg), X) <= 1e-6
        ie.ie_disaggregate(plan.handle, dev(X), r, nrhs)
        assert rel_l2(host(r), oracle.disaggregate(p, X)) <= 1e-6
        ie.ie_near(plan.handle, dev(c), y, nrhs)
        assert rel_l2(host(y), oracle.operator(p, c, "near")) <= 1e-6
        # each column as it is alone
        y1 = empty((1, p.n))
        ie.ie_near(plan.handle, dev(c[-1:]), y1, 1)
        assert rel_l2(host(y1)[0], host(y)[-1]) <= 1e-6
