"""The surrogate's fused training step at widths with remainders: an output width that is no
multiple of 8 (padded rows of the error arrays), rows that are no multiple of a tile, and one Adam
step against its formula on the gradient that npf_mlp_loss_grad returns (the same products)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths,rows", [([5, 16, 32, 13], 129), ([4, 48, 9], 1), ([3, 80, 16, 64], 64)])
def test_one_adam_step(widths, rows):
    from paper_2509_08968_gb300 import build
    build.build()
    from paper_2509_08968_gb300.mlp import Mlp
    from paper_2509_08968_gb300.surrogate import init_weights
    rng = np.random.default_rng(rows)
    W = init_weights(widths, 2, 5)
    X = rng.uniform(-1, 1, (rows, widths[0])).astype(np.float32)
    T = rng.standard_normal((rows, widths[-1])).astype(np.float32)
    lr = 1e-2
    with Mlp(widths, W) as net:
        loss, g = net.loss_grad(X, T)
        hist = net.train(X, T, 1, rows, lr, seed=1)   # one batch: every row, in another order
        got = net.weights().astype(np.float64)
    g = g.astype(np.float64)
    # first step: both moments' bias corrections cancel, w - lr g / (|g| + eps)
    want = W.astype(np.float64) - lr * g / (np.abs(g) + 1e-8)
    # rows in another order move a gradient by FP32 rounding of its sums (at most `rows` terms of
    # 2^-24 of the largest); where that is not small against |g| + eps the step's sign is free
    shift = rows * 2.0 ** -24 * np.abs(g).max()
    sure = np.abs(g) > 1e3 * shift
    assert np.abs(got - want)[sure].max() < lr * 3e-3
    assert np.abs(got - W).max() <= lr * 1.001
    assert abs(hist[0] - loss.mean()) < 1e-5 * loss.mean()
