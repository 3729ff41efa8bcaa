"""Training at the edges of its register tiles: hidden widths around the rows a thread owns
(1, 16, 17, 49, 64).  Adam's first step moves each real and imaginary part that has a gradient, by
the step size at most (the cosine decay starts at lr), so a missing entry shows as a weight that
did not move; read-back and loading are exact inverses;
training lowers e^u."""
import numpy as np
import pytest

import paper_2501_04684_gb300 as ie
import workloads as W

pytestmark = pytest.mark.gpu


def _train(plan, steps, lr):
    ie.ie_cvfcnn_train(plan.handle, ie.cvfcnn_train_opts(max_steps=steps, minibatches=2, eval_every=0, lr=lr, tol=1e-9,
                                                         seed=7))
    return ie.ie_cvfcnn_get_weights(plan.handle)


@pytest.mark.parametrize("hidden", [1, 16, 17, 49, 64])
def test_loss_falls_and_weights_round_trip(hidden):
    p = W.Problem(name="t", G=3, box_ijk=np.array([(0, 0, 0), (2, 0, 0), (2, 2, 1)], dtype=np.int32),
                  nb=np.array([4, 4, 4], dtype=np.int32), P=W.random_P(W.rng(800), np.array([4, 4, 4])), alpha=1.0)
    mask = ie.precmask(ie.IE_PREC_CVFCNN_FP32)
    with ie.Plan(ie.problem_from(p, mask, symmetry=1, cvfcnn_hidden=hidden)) as plan:
        blocks = ie.ie_plan_blocks(plan.handle)
        w0 = _train(plan, 0, 1e-3)
        w1 = _train(plan, 1, 1e-3)
        assert w0[0].shape == (len(blocks), hidden, 192) and w0[2].shape == (len(blocks), 192, hidden)
        # Adam's first step is lr g / (|g| + eps): every part with a gradient moves, by lr at most
        # (and one rounding of the weight)
        d1 = (w1[0] - w0[0]).view(np.float32)
        moved = np.abs(d1) > 0
        assert moved.mean() > 0.9
        assert np.abs(d1).max() <= 1e-3 + np.spacing(np.abs(w1[0]).max())
        # read back, loaded again and read back: the same numbers
        ie.ie_cvfcnn_set_weights(plan.handle, *w1)
        for a, b in zip(w1, ie.ie_cvfcnn_get_weights(plan.handle)):
            assert np.array_equal(a, b)
        info = ie.ie_cvfcnn_train(plan.handle, ie.cvfcnn_train_opts(max_steps=1, minibatches=4, eval_every=0, tol=1e-9))
        late = ie.ie_cvfcnn_train(plan.handle, ie.cvfcnn_train_opts(max_steps=300, minibatches=4, eval_every=0, tol=1e-9))
        assert late["eu_max"] < info["eu_max"]
