"""GPU parity of the far product evaluated as a lattice convolution, against the FP64
brute-force oracle: every transform length on every axis (with the largest extent it serves
and the smallest that needs it), several classes and uneven right-hand-side counts in one
plan, arbitrary box orders, and the columns a scatterer does not have.

Bounds.  Plain products: the framework's 1e-6 relative L2.  A far part read off as the
difference of a full and a near product carries both products' FP32 rounding, so its bound is
1e-6 of the full product.  FP16X3 far products: 2e-6, BF16X3: 5e-5 (the split arithmetic that
takes the adjacent pairs off)."""
import numpy as np
import pytest

import oracle
import paper_2501_04684_gb300 as ie
import workloads as W
from gpu_util import dev, empty, host, rel_l2

pytestmark = pytest.mark.gpu
BOUND = {ie.IE_PREC_FP32: 1e-6, ie.IE_PREC_FP16X3: 2e-6, ie.IE_PREC_BF16X3: 5e-5}
PRECS = list(BOUND)


def _problem(extent, count, seed, nb=(1, 40), identity=False):
    """`count` random boxes (all of them where there are fewer) spanning `extent`, in random order."""
    g = W.rng(seed)
    cells = np.stack(np.meshgrid(*[np.arange(e) for e in extent], indexing="ij"), -1).reshape(-1, 3)
    far = [0, len(cells) - 1]
    rest = g.permutation(np.arange(1, len(cells) - 1))[:max(0, count - 2)]
    ijk = cells[g.permutation(np.concatenate([far, rest]))].astype(np.int32) - 3
    counts = g.integers(nb[0], nb[1] + 1, len(ijk)).astype(np.int32)
    if identity:
        counts[:] = W.NU
    P = None if identity else W.random_P(g, counts)
    return W.Problem(name="conv", G=8, box_ijk=ijk, nb=counts, P=P, alpha=3.0e6)


def _uses(plan, which, prec, nrhs=1):
    return ie.ie_plan_far_bytes(plan.handle, which, prec, nrhs) > 0


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("long", [3, 4, 5, 6, 7, 8, 9, 12, 13, 16, 17, 24, 25, 32, 33, 48, 49, 64])
def test_full_product_at_every_transform_length(long, axis):
    extent = np.roll([long, 2, 3], axis)
    p = _problem(extent, 24, 700 + 3 * long + axis)
    c = W.coefficients(p, 2, 701)
    full, far = oracle.operator(p, c, "full"), oracle.far_matvec(p, c)
    with ie.Plan(ie.problem_from(p, ie.precmask(ie.IE_PREC_FP32), 2)) as plan:
        assert _uses(plan, ie.IE_FULL, ie.IE_PREC_FP32)
        y, yn = empty((2, p.n)), empty((2, p.n))
        ie.ie_matvec(plan.handle, ie.IE_FULL, ie.IE_PREC_FP32, dev(c), y, 2)
        ie.ie_near(plan.handle, dev(c), yn, 2)
        got = host(y)
        assert rel_l2(got, full) <= 1e-6
        assert np.linalg.norm(got - host(yn) - far) <= 1e-6 * np.linalg.norm(full)


@pytest.mark.parametrize("extent,count,identity", [((5, 6, 4), 120, False), ((16, 3, 9), 130, False),
                                                   ((2, 33, 5), 110, True), ((12, 4, 17), 105, False)])
@pytest.mark.parametrize("symmetry", [0, 1])
def test_far_products_and_translations(extent, count, identity, symmetry):
    """Enough far pairs that far products take it too, and their adjacent pairs come off."""
    p = _problem(extent, count, 720 + sum(extent), identity=identity)
    c = W.coefficients(p, 3, 721)
    ref = oracle.far_matvec(p, c)
    X = oracle.aggregate(p, c)
    Yr = oracle.dipole_field(p, X, oracle.FAR)
    with ie.Plan(ie.problem_from(p, ie.precmask(*PRECS), 3, symmetry=symmetry)) as plan:
        for prec in PRECS:
            assert _uses(plan, ie.IE_FAR, prec, 3)
            y, Y = empty((3, p.n)), empty((3, p.n_boxes, W.NU))
            ie.ie_matvec(plan.handle, ie.IE_FAR, prec, dev(c), y, 3)
            assert rel_l2(host(y), ref) <= BOUND[prec], ie.PREC_NAMES[prec]
            ie.ie_translate(plan.handle, prec, dev(X), Y, 3)
            assert rel_l2(host(Y), Yr) <= BOUND[prec], ie.PREC_NAMES[prec]


def test_box_itself_left_out_and_no_adjacent_boxes():
    """self_box_mode = 1 with every second cell occupied: no near block is stored at all."""
    p = _problem((5, 5, 5), 125, 730)
    keep = np.all((p.box_ijk + 3) % 2 == 0, axis=1)
    first = np.repeat(keep, p.nb)
    p = W.Problem(name="sparse", G=8, box_ijk=p.box_ijk[keep], nb=p.nb[keep], P=p.P[first], alpha=2.0, self_box_mode=1)
    c = W.coefficients(p, 1, 731)
    with ie.Plan(ie.problem_from(p, ie.precmask(ie.IE_PREC_FP32))) as plan:
        assert plan.stats["n_near_pairs"] == 0 and _uses(plan, ie.IE_FULL, ie.IE_PREC_FP32)
        y = empty((1, p.n))
        ie.ie_matvec(plan.handle, ie.IE_FULL, ie.IE_PREC_FP32, dev(c), y, 1)
        assert rel_l2(host(y), oracle.operator(p, c, "full")) <= 1e-6


@pytest.mark.parametrize("prec", PRECS, ids=lambda q: ie.PREC_NAMES[q])
def test_batch_of_several_sizes_with_their_own_right_hand_sides(prec):
    """Scatterers of different transform lengths; columns a scatterer does not have get the
    near part of every site pair and no far part, whatever their inputs hold."""
    members = [_problem((4, 4, 4), 64, 740), _problem((7, 3, 5), 60, 741), _problem((4, 4, 4), 50, 742),
               _problem((13, 2, 2), 30, 743)]
    nr = [3, 1, 2, 3]
    b = W.Batch(name="b", G=8, members=members, nrhs=nr, khat=None, pol=None)
    cs = [W.coefficients(m, 3, 744 + i) for i, m in enumerate(members)]
    packed = np.concatenate(cs, axis=1)
    with ie.Plan(ie.problem_from_batch(b, ie.precmask(prec), max_rhs=3, exact_rhs=True)) as plan:
        for which, name in ((ie.IE_FULL, "full"), (ie.IE_FAR, "far")):
            assert _uses(plan, which, prec, 3) or which == ie.IE_FAR
            y = empty((3, b.n))
            ie.ie_matvec(plan.handle, which, prec, dev(packed), y, 3)
            for m, c, q, got in zip(members, cs, nr, b.split(host(y))):
                assert rel_l2(got[:q], oracle.operator(m, c[:q], name)) <= BOUND[prec]
                if q < 3 and which == ie.IE_FULL:
                    assert rel_l2(got[q:], oracle.operator(m, c[q:], "near")) <= 1e-6
                elif q < 3:
                    assert not np.any(got[q:])


def test_where_the_block_products_stay():
    """Low-frequency boxes (the radiative part is far below FP32 rounding of the field), few
    far pairs, boxes scattered over a wide grid and the single-product forms."""
    tiny = W.tiny()
    mask = ie.precmask(*PRECS, ie.IE_PREC_FP16X1)
    with ie.Plan(ie.problem_from(tiny, mask)) as plan:
        assert _uses(plan, ie.IE_FULL, ie.IE_PREC_FP32)
        assert not any(_uses(plan, ie.IE_FAR, q) for q in PRECS)
        assert not _uses(plan, ie.IE_FULL, ie.IE_PREC_FP16X1)
    with ie.Plan(ie.problem_from(W.lfb(tiny, "lfb256"), mask)) as plan:
        assert not any(_uses(plan, ie.IE_FULL, q) for q in PRECS)
    for extent in ((64, 64, 64), (65, 2, 2)):
        with ie.Plan(ie.problem_from(_problem(extent, 20, 750), mask)) as plan:
            assert not any(_uses(plan, ie.IE_FULL, q) for q in PRECS)
