"""Totals of FP32 partial sums near the end of FP32's range: partial sums that are in range add
up as they would in FP64.  A total that leaves the range is infinite, not NaN, and one that leaves
it on the way and comes back is the finite sum (bound: the framework's 1e-6).  Mapping (runs of
16 functions), near product (a block's columns) and near blocks (32 dipole terms)."""
import numpy as np
import pytest

import oracle
import paper_2501_04684_gb300 as ie
import workloads as W
from gpu_util import dev, empty, host, plan_for

pytestmark = pytest.mark.gpu
BIG = 2.5e38


@pytest.mark.parametrize("nrhs", [1, 2, 4])
def test_mapping(nrhs):
    nb = np.full(2, 48, np.int32)
    p = W.Problem(name="big", G=4, box_ijk=np.array([(0, 0, 0), (3, 0, 0)], np.int32), nb=nb,
                  P=np.ones((96, W.NU), np.complex128), alpha=1.0)
    c = np.zeros((nrhs, p.n), np.complex128)
    c[0, [0, 16, 32]] = BIG, BIG, -BIG                # box 0: out of range after two runs, back after three
    c[0, [48, 64]] = BIG                              # box 1: out of range
    with plan_for(p, max_rhs=nrhs) as plan:
        X = empty((nrhs, 2, W.NU))
        ie.ie_aggregate(plan.handle, dev(c), X, nrhs)
        X = host(X)
    assert np.all(np.abs(X[0, 0] - BIG) <= 1e-6 * BIG)
    assert np.all(np.isposinf(X[0, 1].real)) and not np.any(X[0, 1].imag)
    assert not np.any(X[1:])


@pytest.mark.parametrize("nb", [1, 40, 70])
def test_near_product(nb):
    """The centre of 3^3 boxes: blocks 0, 8, 16 and 24 of its row are one warp's, in that order."""
    g = W.rng(970)
    counts = np.full(27, nb, np.int32)
    p = W.Problem(name="big", G=3, box_ijk=W.full_grid(3), nb=counts, P=W.random_P(g, counts), alpha=0.0)
    centre = int(np.flatnonzero((p.box_ijk == 1).all(1))[0])
    order = [int(np.flatnonzero((p.box_ijk == (1 - ex, 1 - ey, 1 - ez)).all(1))[0])
             for ex in (-1, 0, 1) for ey in (-1, 0, 1) for ez in (-1, 0, 1)]
    row = centre * nb
    with plan_for(p) as plan:
        def near(c):
            y = empty((1, p.n))
            ie.ie_near(plan.handle, dev(c), y, 1)
            return host(y)[0, row]
        for signs, want in (((1, 1, -1), BIG), ((1, 1, 0), np.inf)):
            c = np.zeros((1, p.n), np.complex128)
            for s, k in zip(signs, (0, 8, 16)):
                e = np.zeros((1, p.n), np.complex128)
                e[0, order[k] * nb] = 1
                N = near(e)
                assert abs(N) > 10                    # so that c stays in range
                c[0, order[k] * nb] = s * BIG / N
            y = near(c)
            if np.isinf(want):
                assert np.isposinf(y.real) and np.isfinite(y.imag)
            else:
                assert abs(y - want) <= 4e-6 * want   # each coefficient carries one rounding, sums of 3 BIG


def test_near_blocks():
    """One box: W = G P^T gets three terms from different runs of 32 whose first two leave the range
    in some row and whose sum is in range in every row; N = P W has to be finite and right."""
    p = W.Problem(name="big", G=1, box_ijk=np.zeros((1, 3), np.int32), nb=np.array([2], np.int32), P=None, alpha=0.0)
    G = oracle.coupling_block(p, np.zeros(3, np.int32))
    # y moments of the neighbours of site 9 along y (sites 5 and 13: the largest entries of G, one
    # sign) and along z (site 25: the other sign); 16, 40 and 76 lie in three runs
    at, w, big = np.array([16, 40, 76]), np.ones(3), 3.0e38
    t = G[:, at] * w

    def parts(a):
        return max(np.abs(a.real).max(), np.abs(a.imag).max())
    inside = max(max(parts(t[:, i]) for i in range(3)), parts(t.sum(1)))
    assert parts(t[:, 0] + t[:, 1]) > 1.25 * inside
    w = w * big / inside                          # every term and total within 3e38, the way above 3.7e38
    P = np.zeros((2, W.NU), np.complex128)
    P[0, at] = w
    P[1, ::7] = 1e-36
    p.P = P
    want = (P[1].astype(np.complex64).astype(np.complex128) @ G @ P[0].astype(np.complex64).astype(np.complex128))
    with plan_for(p) as plan:
        y = empty((1, 2))
        ie.ie_near(plan.handle, dev(np.array([[1.0, 0.0]])), y, 1)
        got = host(y)[0, 1]
    assert abs(got - want) <= 1e-5 * (np.abs(P[1]) @ np.abs(G) @ np.abs(P[0]))
