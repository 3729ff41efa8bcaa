"""The two forms of a far product, each asserted to be the one that runs (ie_plan_far_bytes).

Convolution: the radiative part of a product at the box edges it serves (real dipole moments on
identity P: Re y = Re(G) x alone), with the bounds of the low-frequency tests, and plans on
several streams and threads.  Block products, which still serve FP32 and FP16X3 at lambda/256:
the symmetric store's packed lists against the full store and the oracle on the 16^3 shell, and
the shared store's blocks."""
import threading

import numpy as np
import pytest
import torch

import oracle
import paper_2501_04684_gb300 as ie
import workloads as W
from gpu_util import dev, empty, host, rel_l2

pytestmark = pytest.mark.gpu
BOUND = {ie.IE_PREC_FP32: 1e-6, ie.IE_PREC_BF16X3: 5e-5, ie.IE_PREC_FP16X3: 2e-6}
PRECS = list(BOUND)


def _conv(plan, which, prec, nrhs=1):
    return ie.ie_plan_far_bytes(plan.handle, which, prec, nrhs) > 0


def _low_shell():
    p = W.lfb(W.shell16(), "lfb256")
    p.alpha = W.alpha_for(p.name)
    return p


@pytest.mark.parametrize("edge", [4.0, 8.0])
@pytest.mark.parametrize("which,name", [(ie.IE_FAR, "far"), (ie.IE_FULL, "full")], ids=["far", "full"])
def test_radiative_part_of_a_convolution(edge, which, name):
    ijk = W.full_grid(6)
    p = W.Problem(name="radiative", G=6, box_ijk=ijk, nb=np.full(len(ijk), W.NU, np.int32), P=None, alpha=0.0, a=1.0 / edge)
    c = W.rng(1100).standard_normal((1, p.n)).astype(np.complex128)
    ref = oracle.operator(p, c.astype(np.complex64).astype(np.complex128), name)
    with ie.Plan(ie.problem_from(p, ie.precmask(*PRECS))) as plan:
        for prec in PRECS:
            assert _conv(plan, which, prec)
            y = empty((1, p.n))
            ie.ie_matvec(plan.handle, which, prec, dev(c), y, 1)
            got = host(y)
            for part in (np.real, np.imag):
                assert rel_l2(part(got), part(ref)) <= BOUND[prec], (ie.PREC_NAMES[prec], part.__name__)


def test_symmetric_and_full_store_blocks_on_the_shell():
    p = _low_shell()
    c = W.coefficients(p, 1, W.SEED_C["shell16"])
    targets = W.subsample_boxes(p, 12, W.SEED_SUBSAMPLE["shell16"])
    rows = oracle.basis_rows(p, targets)
    ref = oracle.far_matvec(p, c, targets=targets)
    out = {}
    for sym in (0, 1):
        with ie.Plan(ie.problem_from(p, ie.precmask(ie.IE_PREC_FP32, ie.IE_PREC_FP16X3), symmetry=sym)) as plan:
            for prec in (ie.IE_PREC_FP32, ie.IE_PREC_FP16X3):
                assert not _conv(plan, ie.IE_FAR, prec)
                y = empty((1, p.n))
                ie.ie_matvec(plan.handle, ie.IE_FAR, prec, dev(c), y, 1)
                out[sym, prec] = host(y)
                assert rel_l2(out[sym, prec][:, rows], ref) <= BOUND[prec]
    for prec in (ie.IE_PREC_FP32, ie.IE_PREC_FP16X3):
        assert rel_l2(out[1, prec], out[0, prec]) <= BOUND[prec]


def _spec(p, precs):
    return ie.store_spec(p.k, p.eta, p.a, 15, ie.precmask(*precs))


@pytest.mark.parametrize("prec", [ie.IE_PREC_FP32, ie.IE_PREC_FP16X3], ids=lambda q: ie.PREC_NAMES[q])
def test_shared_store_blocks(prec):
    """A plan on a store reads the store's blocks, also after its creator has released it."""
    p = _low_shell()
    c = dev(W.coefficients(p, 1, 1110))
    pr = ie.problem_from(p, ie.precmask(prec), symmetry=1)
    store = ie.Store(_spec(p, [prec]))
    out = []
    with ie.Plan(pr, store=store) as plan, ie.Plan(pr) as own:
        for released in (False, True):
            if released:
                store.close()
            for pl in (plan, own):
                assert not _conv(pl, ie.IE_FULL, prec)
                y = empty((1, p.n))
                ie.ie_matvec(pl.handle, ie.IE_FULL, prec, c, y, 1)
                out.append(host(y))
    assert rel_l2(out[0], out[1]) <= 1e-6 and rel_l2(out[2], out[3]) <= 1e-6


def test_plans_on_several_streams_and_threads():
    """Each plan has its own side stream: full and far products of two plans, interleaved on two
    streams and then from a thread each, give what each plan gives alone."""
    probs = []
    for k, n in enumerate((5, 6)):
        g = W.rng(1120 + k)
        ijk = W.full_grid(n)
        nb = np.full(len(ijk), 12, np.int32)
        probs.append(W.Problem(name="s", G=n, box_ijk=ijk, nb=nb, P=W.random_P(g, nb), alpha=4e6))
    prec = ie.IE_PREC_FP16X3
    plans = [ie.Plan(ie.problem_from(p, ie.precmask(prec), 2, symmetry=1)) for p in probs]
    try:
        xs = [dev(W.coefficients(p, 2, 1122 + k)) for k, p in enumerate(probs)]
        alone = []
        for p, plan, x in zip(probs, plans, xs):
            assert _conv(plan, ie.IE_FAR, prec, 2)
            for which in (ie.IE_FULL, ie.IE_FAR):
                y = empty((2, p.n))
                ie.ie_matvec(plan.handle, which, prec, x, y, 2)
                alone.append(host(y))
        streams = [torch.cuda.Stream(), torch.cuda.Stream()]
        ys = [[empty((2, p.n)) for _ in range(2)] for p in probs]
        torch.cuda.synchronize()
        errs = []

        def check():
            torch.cuda.synchronize()
            for k in range(2):
                assert rel_l2(host(ys[k][0]), alone[2 * k]) <= 1e-6
                assert rel_l2(host(ys[k][1]), alone[2 * k + 1]) <= 2e-6

        def queue(k, times):
            try:
                for _ in range(times):
                    ie.ie_matvec(plans[k].handle, ie.IE_FULL, prec, xs[k], ys[k][0], 2, streams[k])
                    ie.ie_matvec(plans[k].handle, ie.IE_FAR, prec, xs[k], ys[k][1], 2, streams[k])
            except Exception as e:      # surfaced below
                errs.append(e)
        for _ in range(20):
            queue(0, 1)
            queue(1, 1)
        check()
        ts = [threading.Thread(target=queue, args=(k, 30)) for k in range(2)]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
        assert not errs, errs
        check()
    finally:
        for plan in plans:
            plan.close()
