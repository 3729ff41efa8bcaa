"""Far products and translations of uneven inputs, box by box.  A transform rounds relative to
the scatterer's whole field, a block product relative to what reaches a box; where an input's
far sources are weak beside a box's own neighbourhood only the second keeps that box's digits,
keeps the neighbourhood of a lone source at exactly zero and keeps a non-finite value away from
boxes that it is not far from.

Bounds, per target box: the framework's bounds of a whole product (1e-6 FP32, 2e-6 FP16X3, 5e-5
BF16X3) times 4: a factor 2 for the worst box beside the whole vector, and a factor 2 for the
unevenness that the convolution is used up to (sources' energy at most 4 times the far one's;
rounding grows with its square root)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2501_04684_gb300 as ie
import workloads as W
from gpu_util import dev, empty, host

pytestmark = pytest.mark.gpu
BOUND = {ie.IE_PREC_FP32: 4e-6, ie.IE_PREC_FP16X3: 8e-6, ie.IE_PREC_BF16X3: 2e-4}
PRECS = list(BOUND)
NAMES = dict(ids=lambda q: ie.PREC_NAMES[q])


def _cube(n, seed):
    g = W.rng(seed)
    ijk = W.full_grid(n)[g.permutation(n ** 3)]
    nb = g.integers(4, 13, len(ijk)).astype(np.int32)
    return W.Problem(name="uneven", G=n, box_ijk=ijk, nb=nb, P=W.random_P(g, nb), alpha=1.0)


def _rows(p, b):
    return slice(p.offsets[b], p.offsets[b + 1])


def _box_errors(p, got, ref):
    return np.array([np.linalg.norm(got[_rows(p, b)] - ref[_rows(p, b)]) / np.linalg.norm(ref[_rows(p, b)])
                     for b in range(p.n_boxes)])


def _near(p, b):
    return np.abs(p.box_ijk - p.box_ijk[b]).max(1) <= 1


def _far(plan, prec, c):
    y = empty(c.shape)
    ie.ie_matvec(plan.handle, ie.IE_FAR, prec, dev(c), y, c.shape[0])
    return host(y)


def _translate(plan, prec, X):
    Y = empty(X.shape)
    ie.ie_translate(plan.handle, prec, dev(X), Y, X.shape[0])
    return host(Y)


@pytest.mark.parametrize("symmetry", [0, 1])
@pytest.mark.parametrize("prec", PRECS, **NAMES)
def test_one_box_above_the_rest(prec, symmetry):
    p = _cube(6, 900)
    strong = 77
    with ie.Plan(ie.problem_from(p, ie.precmask(prec), 2, symmetry=symmetry)) as plan:
        assert ie.ie_plan_far_bytes(plan.handle, ie.IE_FAR, prec, 2) > 0
        for scale in (1.0, 10.0, 30.0, 1e2, 1e4, 1e6):      # 30 is about where the forms change
            c = W.coefficients(p, 2, 901)
            c[1, _rows(p, strong)] *= scale                  # the other column stays even
            got, ref = _far(plan, prec, c), oracle.far_matvec(p, c.astype(np.complex64))
            for r in range(2):
                assert _box_errors(p, got[r], ref[r]).max() <= BOUND[prec], (scale, r)


@pytest.mark.parametrize("scale", [1.0, 1e3, 1e6, 0.0])
def test_full_products_box_by_box(scale):
    """One box `scale` above the rest, or (0) alone: the near part holds what a box is near to."""
    p = _cube(6, 905)
    c = W.coefficients(p, 1, 906)
    if scale:
        c[0, _rows(p, 31)] *= scale
    else:
        c[0, :p.offsets[31]] = c[0, p.offsets[32]:] = 0
    with ie.Plan(ie.problem_from(p, ie.precmask(ie.IE_PREC_FP32))) as plan:
        assert ie.ie_plan_far_bytes(plan.handle, ie.IE_FULL, ie.IE_PREC_FP32, 1) > 0
        y = empty((1, p.n))
        ie.ie_matvec(plan.handle, ie.IE_FULL, ie.IE_PREC_FP32, dev(c), y, 1)
        got = host(y)[0]
    assert _box_errors(p, got, oracle.operator(p, c.astype(np.complex64), "full")[0]).max() <= BOUND[ie.IE_PREC_FP32]


@pytest.mark.parametrize("prec", PRECS, **NAMES)
def test_a_lone_source_leaves_its_neighbourhood_at_zero(prec):
    p = _cube(6, 910)
    one = int(np.flatnonzero((p.box_ijk == (2, 3, 2)).all(1))[0])
    X = np.zeros((1, p.n_boxes, W.NU), np.complex128)
    X[0, one] = W.complex_normal(W.rng(911), W.NU)
    ref = oracle.dipole_field(p, X.astype(np.complex64), oracle.FAR)[0]
    near = _near(p, one)
    assert near.sum() == 27 and not np.any(ref[near])
    with ie.Plan(ie.problem_from(p, ie.precmask(prec))) as plan:
        assert ie.ie_plan_far_bytes(plan.handle, ie.IE_FAR, prec, 1) > 0
        got = _translate(plan, prec, X)[0]
    assert not np.any(got[near])
    err = np.linalg.norm(got[~near] - ref[~near], axis=1) / np.linalg.norm(ref[~near], axis=1)
    assert err.max() <= BOUND[prec]


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf], ids=["nan", "inf", "-inf"])
@pytest.mark.parametrize("prec", [ie.IE_PREC_FP32, ie.IE_PREC_BF16X3], **NAMES)
def test_a_non_finite_value_stays_with_the_boxes_it_is_far_from(prec, value):
    p = _cube(6, 920)
    bad = int(np.flatnonzero((p.box_ijk == (1, 2, 3)).all(1))[0])
    X = W.complex_normal(W.rng(921), (2, p.n_boxes, W.NU))
    X[0, bad, 5] = value
    clean = X.copy()
    clean[0, bad] = 0
    ref = oracle.dipole_field(p, clean.astype(np.complex64), oracle.FAR)
    near = _near(p, bad)
    with ie.Plan(ie.problem_from(p, ie.precmask(prec), 2)) as plan:
        got = _translate(plan, prec, X)
    err = np.linalg.norm(got - ref, axis=2) / np.linalg.norm(ref, axis=2)
    assert err[0, near].max() <= BOUND[prec] and err[1].max() <= BOUND[prec]
    assert not np.isfinite(got[0, ~near]).all(axis=1).any()


@pytest.mark.parametrize("scale", [1e-34, 1e30])
def test_amplitudes_at_the_ends_of_the_range(scale):
    p = _cube(5, 930)
    X = W.complex_normal(W.rng(931), (1, p.n_boxes, W.NU)) * scale
    ref = oracle.dipole_field(p, X.astype(np.complex64), oracle.FAR)[0]
    with ie.Plan(ie.problem_from(p, ie.precmask(ie.IE_PREC_FP32))) as plan:
        got = _translate(plan, ie.IE_PREC_FP32, X)[0]
    assert (np.linalg.norm(got - ref, axis=1) / np.linalg.norm(ref, axis=1)).max() <= BOUND[ie.IE_PREC_FP32]


def test_one_scatterer_of_a_batch_uneven_in_one_of_its_columns():
    members = [_cube(5, 940), _cube(4, 941), _cube(5, 942)]
    nr = [2, 3, 1]
    b = W.Batch(name="b", G=5, members=members, nrhs=nr, khat=None, pol=None)
    cs = [W.coefficients(m, 3, 943 + i) for i, m in enumerate(members)]
    for m, c, q in zip(members, cs, nr):
        c[q:] = 0
    with ie.Plan(ie.problem_from_batch(b, ie.precmask(ie.IE_PREC_FP16X3), max_rhs=3, exact_rhs=True)) as plan:
        assert ie.ie_plan_far_bytes(plan.handle, ie.IE_FAR, ie.IE_PREC_FP16X3, 3) > 0
        for scale in (1.0, 1e5):
            cs[1][2, _rows(members[1], 9)] *= scale
            got = _far(plan, ie.IE_PREC_FP16X3, np.concatenate(cs, axis=1))
            for m, c, q, y in zip(members, cs, nr, b.split(got)):
                ref = oracle.far_matvec(m, c[:q].astype(np.complex64))
                for r in range(q):
                    assert _box_errors(m, y[r], ref[r]).max() <= BOUND[ie.IE_PREC_FP16X3], (scale, r)
                assert not np.any(y[q:])


@pytest.mark.parametrize("extent", [(3, 3, 40), (1, 1, 110)])
def test_boxes_without_far_partners_get_zero(extent):
    """A small scatterer beside one large enough for the convolution: nothing is far from its boxes."""
    g = W.rng(950)
    cells = np.stack(np.meshgrid(*[np.arange(e) for e in extent], indexing="ij"), -1).reshape(-1, 3)[:340].astype(np.int32)
    small = W.full_grid(2)
    ijk = np.concatenate([cells, small])
    nb = np.full(len(ijk), 6, np.int32)
    group = np.array([0] * len(cells) + [1] * len(small), np.int32)
    P = W.random_P(g, nb)
    big = W.Problem(name="big", G=40, box_ijk=cells, nb=nb[:len(cells)], P=P[:6 * len(cells)], alpha=1.0)
    c = W.complex_normal(g, (1, 6 * len(ijk)))
    pr = ie.make_problem(big.k, big.eta, big.a, 40, ijk, nb, P, 1.0, ie.precmask(ie.IE_PREC_FP32), 1, box_group=group,
                         group_alpha=np.ones(2))
    with ie.Plan(pr) as plan:
        got = _far(plan, ie.IE_PREC_FP32, c)[0]
    ref = oracle.far_matvec(big, c[:, :big.n].astype(np.complex64))[0]
    assert not np.any(got[big.n:])
    assert _box_errors(big, got[:big.n], ref).max() <= BOUND[ie.IE_PREC_FP32]


def test_a_captured_product_follows_its_input():
    p = _cube(6, 960)
    c = W.coefficients(p, 1, 961)
    with ie.Plan(ie.problem_from(p, ie.precmask(ie.IE_PREC_FP16X3))) as plan:
        x, y = dev(c), empty((1, p.n))
        ie.ie_matvec(plan.handle, ie.IE_FAR, ie.IE_PREC_FP16X3, x, y, 1)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            ie.ie_matvec(plan.handle, ie.IE_FAR, ie.IE_PREC_FP16X3, x, y, 1)
        for scale in (1.0, 1e5, 1e-5, 1.0):
            q = c.copy()
            q[0, _rows(p, 100)] *= scale
            x.copy_(dev(q))
            graph.replay()
            ref = oracle.far_matvec(p, q.astype(np.complex64))[0]
            assert _box_errors(p, host(y)[0], ref).max() <= BOUND[ie.IE_PREC_FP16X3], scale
