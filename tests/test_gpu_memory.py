"""Device memory of solvers."""
import numpy as np
import pytest

import paper_2501_04684_gb300 as ie
import workloads as W

pytestmark = pytest.mark.gpu


def _problem(n, nb, edge=4.0):
    g = W.rng(1000 + n)
    ijk = W.full_grid(n)
    counts = np.full(len(ijk), nb, np.int32)
    return W.Problem(name="memory", G=n, box_ijk=ijk, nb=counts, P=W.random_P(g, counts), alpha=W.alpha_for("tiny"), a=1.0 / edge)


def test_solver_footprint_counts_the_refinement():
    """A refined solve keeps, per unknown and column, an FP64 iterate and three FP32 vectors (40
    bytes), and one FP64 pair per chunk of 512 unknowns."""
    p, R = _problem(4, 20), 3
    with ie.Plan(ie.problem_from(p, ie.precmask(ie.IE_PREC_FP32), R)) as plan:
        plain = ie.ie_solver_footprint(plan.handle, R, ie.solve_opts())
        refined = ie.ie_solver_footprint(plan.handle, R, ie.solve_opts(refine=1))
        assert refined - plain == 40 * R * p.n + 16 * R * -(-p.n // 512)
