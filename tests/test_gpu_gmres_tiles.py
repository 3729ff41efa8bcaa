"""GMRES at the edges of its kernels' tiles: restart lengths around the groups of four Krylov
vectors the dot products take together, systems shorter and longer than a chunk of 512
unknowns, and a batch in which a scatterer has no boxes.  Bounds: the recomputed residual
within the requested tolerance (the recurrence stops there; FP32 products add 1e-6), against
the FP64 oracle's operator."""
import numpy as np
import pytest

import oracle
import paper_2501_04684_gb300 as ie
import workloads as W
from gpu_util import dev, empty, host

pytestmark = pytest.mark.gpu


def _problem(boxes, nb, seed):
    g = W.rng(seed)
    ijk = W.full_grid(3)[:boxes]
    counts = np.full(len(ijk), nb, dtype=np.int32)
    p = W.Problem(name="g", G=3, box_ijk=ijk, nb=counts, P=W.random_P(g, counts), alpha=0.0)
    p.alpha = W.alpha_for("tiny")
    return p


def _residual(p, x, v):
    return np.linalg.norm(oracle.operator(p, x, "full") - v, axis=1) / np.linalg.norm(v, axis=1)


@pytest.mark.parametrize("restart", [1, 3, 4, 5, 8, 9, 64])
@pytest.mark.parametrize("boxes,nb", [(2, 5), (27, 38)])
def test_restart_lengths(restart, boxes, nb):
    p = _problem(boxes, nb, 780 + boxes)
    v = W.coefficients(p, 3, 781) * np.array([[1.0], [1e-3], [1e3]])
    with ie.Plan(ie.problem_from(p, ie.precmask(ie.IE_PREC_FP32), 3)) as plan:
        x = empty((3, p.n))
        st, info = ie.ie_solve(plan.handle, dev(v), x, 3, ie.solve_opts(tol=1e-6, restart=restart, max_iters=2000))
        assert st == ie.IE_OK and info["converged"] == 1 and info["relres"] <= 1e-6
        assert np.all(_residual(p, host(x), v.astype(np.complex64)) <= 2e-6)
        # a zero right-hand side beside the others ends at once with a zero solution
        v[1] = 0
        st, info = ie.ie_solve(plan.handle, dev(v), x, 3, ie.solve_opts(tol=1e-6, restart=restart, max_iters=2000))
        assert st == ie.IE_OK and not np.any(host(x)[1])


def test_refined_solves_repeat_and_move():
    """The refinement's kept buffers: repeated calls, another right-hand side, other tensors."""
    p = _problem(27, 20, 785)
    precs = [ie.IE_PREC_FP32, ie.IE_PREC_FP16X1, ie.IE_PREC_FP16X3]
    with ie.Plan(ie.problem_from(p, ie.precmask(*precs), 2)) as plan:
        o = ie.solve_opts(tol=1e-5, prec=ie.IE_PREC_FP16X1, refine=1, refine_prec=ie.IE_PREC_FP16X3, inner_tol=1e-3)
        for seed in (786, 787, 786):
            v = W.coefficients(p, 2, seed)
            x = empty((2, p.n))
            st, info = ie.ie_solve(plan.handle, dev(v), x, 2, o)
            assert st == ie.IE_OK and info["refinements"] >= 1, info
            assert np.all(_residual(p, host(x), v.astype(np.complex64)) <= 1.2e-5)


def test_scatterer_without_boxes():
    a, b = _problem(8, 12, 790), _problem(12, 9, 791)
    ijk = np.concatenate([a.box_ijk, b.box_ijk])
    group = np.array([0] * a.n_boxes + [2] * b.n_boxes, dtype=np.int32)
    al = a.alpha
    pr = ie.make_problem(a.k, a.eta, a.a, 3, ijk, np.concatenate([a.nb, b.nb]), np.concatenate([a.P, b.P]), al,
                         ie.precmask(ie.IE_PREC_FP32), 2, box_group=group, group_alpha=np.full(4, al))
    va, vb = W.coefficients(a, 2, 792), W.coefficients(b, 2, 793)
    with ie.Plan(pr) as plan:
        assert plan.stats["n_groups"] == 4
        x = empty((2, a.n + b.n))
        st, info = ie.ie_solve(plan.handle, dev(np.concatenate([va, vb], axis=1)), x, 2, ie.solve_opts(tol=1e-6))
        assert st == ie.IE_OK and info["converged"] == 1, info
        got = host(x)
    assert np.all(_residual(a, got[:, :a.n], va.astype(np.complex64)) <= 2e-6)
    assert np.all(_residual(b, got[:, a.n:], vb.astype(np.complex64)) <= 2e-6)
