"""The screen's training step at the edges of its tiles (4 rows a block, 256
rows a stage): gradients against the fp64 oracle, and one Adam step, whose
update is -lr g / (|g| + 1e-8) whatever the moments' rounding."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("quantile", [0.0, 0.9])
@pytest.mark.parametrize("n", [1, 3, 4, 5, 255, 256, 257, 513, 4101])
def test_gradient_and_first_step(n, quantile):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_10459_gb300 as idtx
    from paper_1807_10459_gb300 import build
    build.build()
    rng = np.random.default_rng(n)
    sc = idtx.Screen(seed=n)
    sc.params[:] += (rng.standard_normal(sc.params.size) * 0.05).astype(np.float32)
    sc.feat_mean[:] = rng.standard_normal(10).astype(np.float32)
    sc.feat_scale[:] = (0.5 + rng.random(10)).astype(np.float32)
    x = rng.standard_normal((n, 10)).astype(np.float32)
    t = (np.tanh(x[:, 0]) + 0.3 * x[:, 6] * x[:, 8]).astype(np.float32)
    rl, rg = oracle.mlp_loss_grad(sc.params, 10, 64, sc.feat_mean, sc.feat_scale, x, t,
                                  bf16=True, quantile=quantile)
    loss, g = idtx.screen_loss_grad(sc, x, t, quantile=quantile)
    assert abs(loss - rl) <= 1e-5 * max(1.0, rl)
    assert np.max(np.abs(g - rg)) <= 1e-4 * max(1.0, np.max(np.abs(rg)))
    before, lr = sc.params.copy(), 1e-3
    idtx.screen_train(sc, x, t, epochs=1, batch=n, lr=lr, seed=1, quantile=quantile)
    # parameters whose gradient's sign is certain move by lr, up to the
    # rounding of a parameter of at most 4 (2^-22) and of the quotient
    sure = np.abs(rg) > 2e-4 * max(1.0, np.max(np.abs(rg)))
    step = sc.params.astype(np.float64) - before
    assert sure.sum() > 100
    assert np.max(np.abs(step[sure] + lr * np.sign(rg[sure]))) < 1e-6
    # one that no row reaches stays
    assert np.array_equal(sc.params[g == 0], before[g == 0])
