"""One Adam step of the networks' training against the gradient in 64 bits: the inputs and the
initial weights are the kernel's (its counter-based generator is restated here, the weights are
read back).  Adam's first step moves each real and imaginary part by -lr g / (|g| + 1e-8), so
every entry of W1, b1, W2 and b2 with a gradient g above the FP32 rounding of its sum (1e-4 of the
largest; the sums have at most 64 x 192 terms) has to have moved by that, within 1e-2 of lr and
the rounding of the stored weight."""
import numpy as np
import pytest

import oracle
import paper_2501_04684_gb300 as ie
import workloads as W

pytestmark = pytest.mark.gpu
U64 = np.uint64
SEED, BATCH = 11, 32


def _mix(z):
    z = z + U64(0x9E3779B97F4A7C15)
    z = (z ^ (z >> U64(30))) * U64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> U64(27))) * U64(0x94D049BB133111EB)
    return z ^ (z >> U64(31))


def _inputs(net, step):
    """(192, 32) inputs of one minibatch, uniform in [-1, 1)^2, over their largest modulus."""
    with np.errstate(over="ignore"):
        idx = np.arange(BATCH * W.NU, dtype=U64)
        r = _mix(U64(SEED) ^ _mix((U64(net) << U64(32) | U64(step)) ^ _mix(idx)))
    a = (r >> U64(40)).astype(float) / 16777216.0
    b = ((r >> U64(16)) & U64(0xFFFFFF)).astype(float) / 16777216.0
    x = ((2 * a - 1) + 1j * (2 * b - 1)).reshape(BATCH, W.NU).T
    return x / np.abs(x).max(0)


@pytest.mark.parametrize("hidden", [1, 17, 50, 64])
def test_first_step_follows_the_gradient(hidden):
    nb = np.full(3, 4, np.int32)
    p = W.Problem(name="t", G=3, box_ijk=np.array([(0, 0, 0), (2, 0, 0), (2, 2, 1)], np.int32), nb=nb,
                  P=W.random_P(W.rng(1130), nb), alpha=1.0)
    lr, micro = 1e-3, 2
    with ie.Plan(ie.problem_from(p, ie.precmask(ie.IE_PREC_CVFCNN_FP32), symmetry=1, cvfcnn_hidden=hidden)) as plan:
        blocks = ie.ie_plan_blocks(plan.handle)
        state = []
        for steps in (0, 1):
            ie.ie_cvfcnn_train(plan.handle, ie.cvfcnn_train_opts(max_steps=steps, minibatches=micro, eval_every=0, lr=lr,
                                                                 tol=1e-9, seed=SEED))
            state.append([w.astype(np.complex128) for w in ie.ie_cvfcnn_get_weights(plan.handle)])
    for k, d in enumerate(blocks):
        G = oracle.coupling_block(p, d)
        g = np.abs(G).max()                             # the kernel trains G / g; W2 and b2 come back times g
        W1, b1, W2, b2 = (w[k] for w in state[0])
        W2, b2 = W2 / g, b2 / g
        grad = [np.zeros_like(w) for w in (W1, b1, W2, b2)]
        for m in range(micro):
            x = _inputs(k, m)
            z = W1 @ x + b1[:, None]
            h = np.maximum(z.real, 0) + 1j * np.maximum(z.imag, 0)
            r = 2.0 / (BATCH * W.NU) * (W2 @ h + b2[:, None] - G @ x / g)
            dh = W2.conj().T @ r
            dz = np.where(z.real > 0, dh.real, 0) + 1j * np.where(z.imag > 0, dh.imag, 0)
            for q, v in zip(grad, (dz @ x.conj().T, dz.sum(1), r @ h.conj().T, r.sum(1))):
                q += v
        for name, q, w0, w1, unit in zip(("W1", "b1", "W2", "b2"), grad, (w[k] for w in state[0]), (w[k] for w in state[1]),
                                         (1, 1, g, g)):
            for part in (np.real, np.imag):
                gr, move = part(q), part(w1 - w0)
                clear = np.abs(gr) > 1e-4 * np.abs(gr).max()
                assert clear.mean() > 0.5, name
                slack = 1e-2 * lr * unit + 2 * np.spacing(np.float32(np.abs(part(w1)).max()))
                want = -lr * unit * gr / (np.abs(gr) + 1e-8)
                assert np.all(np.abs(move - want)[clear] <= slack), (name, part.__name__, k)
