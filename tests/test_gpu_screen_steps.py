"""Several steps of the screen's training, whose kernels start before the one in
front of them has ended, against a host loop with the oracle's gradients: three
epochs of two full batches and a short one.

The learning rate is large, so that a parameter or moment of the step before, or
rows of another order, would show: the median parameter then ends 0.02 to 0.03
off (the loop with the last step's parameters is run to confirm it).  A relative
error of 1e-6 in every gradient ends 1.5e-4 off in the median (training
amplifies it: a step's size does not depend on the gradient's), so the median
may be 5e-3 off."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPOCHS, BATCH, LR, SEED = 3, 32, 0.02, 5


def _host_loop(sc, x, t, stale=False):
    p = last = sc.params.astype(np.float32)
    m, v, step = np.zeros(p.size), np.zeros(p.size), 0
    for ep in range(EPOCHS):
        order = oracle.perm(SEED, ep, len(t))
        for at in range(0, len(t), BATCH):
            rows = order[at:at + BATCH]
            _, g = oracle.mlp_loss_grad(last if stale else p, 10, 64, sc.feat_mean, sc.feat_scale,
                                        x[rows], t[rows], bf16=True, quantile=0.0)
            step += 1
            m = 0.9 * m + 0.1 * g
            v = 0.999 * v + 0.001 * g * g
            last, p = p, (p - LR * (m / (1 - 0.9 ** step)) /
                          (np.sqrt(v / (1 - 0.999 ** step)) + 1e-8)).astype(np.float32)
    return p


def test_steps_follow_each_other():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_10459_gb300 as idtx
    from paper_1807_10459_gb300 import build
    build.build()
    rng = np.random.default_rng(3)
    sc = idtx.Screen(seed=3)
    x = rng.standard_normal((90, 10)).astype(np.float32)
    t = (np.tanh(x[:, 0]) + 0.3 * x[:, 6] * x[:, 8]).astype(np.float32)
    want, stale = _host_loop(sc, x, t), _host_loop(sc, x, t, stale=True)
    assert np.median(np.abs(stale - want)) > 0.02
    idtx.screen_train(sc, x, t, epochs=EPOCHS, batch=BATCH, lr=LR, seed=SEED, quantile=0.0)
    assert np.median(np.abs(sc.params - want)) < 5e-3
