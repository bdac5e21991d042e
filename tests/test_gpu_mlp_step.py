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


def _fma(a, b, c):
    """a b + c with one rounding to FP32 (long double holds the product exactly)."""
    x = np.longdouble
    return (a.astype(x) * np.asarray(b, x) + c.astype(x)).astype(np.float32)


@pytest.mark.parametrize("widths,rows,scale", [([4, 48, 9], 1, 1.0), ([5, 16, 32, 13], 64, 1.0), ([4, 256, 64], 33, 1.0),
                                               ([4, 48, 9], 3, 1e-14), ([4, 48, 9], 3, 1e-22), ([4, 48, 9], 3, 1e9)])
def test_adam_steps_are_exact(widths, rows, scale):
    """Adam's arithmetic bit for bit: FP32, every operation rounded to nearest, the moments' new terms
    fused with their sums, true divisions (the inputs' scale brings the first layer's moments to the ends
    of the range: squares below 2^-100, below the normal numbers and above 2^50; some weights start at
    zero or next to it, where the smallest update counts). With equal rows the order of a batch does not
    matter, so each step's gradient is npf_mlp_loss_grad's."""
    from paper_2509_08968_gb300 import build
    build.build()
    from paper_2509_08968_gb300.mlp import Mlp
    from paper_2509_08968_gb300.surrogate import init_weights
    rng = np.random.default_rng(7 + rows)
    w = init_weights(widths, 2, 6)
    w[:, ::7] = 0
    w[:, 3::7] *= np.float32(1e-20)
    X = np.repeat((scale * rng.uniform(-1, 1, (1, widths[0]))).astype(np.float32), rows, 0)
    T = np.repeat(rng.standard_normal((1, widths[-1])).astype(np.float32), rows, 0)
    f = np.float32
    b1, b2, one = f(0.9), f(0.999), f(1.0)
    m, v = np.zeros_like(w), np.zeros_like(w)
    with Mlp(widths, w) as net:
        for k in range(1, 13):
            _, g = net.loss_grad(X, T)
            assert (g == 0).any() and (g != 0).any()
            net.train(X, T, 1, rows, 1e-2, seed=k)
            m, v = _fma(g, one - b1, b1 * m), _fma((one - b2) * g, g, b2 * v)
            c1, c2 = f(1.0 - float(b1) ** k), f(1.0 - float(b2) ** k)
            w = w - f(1e-2) * (m / c1) / (np.sqrt(v / c2) + f(1e-8))
            got = net.weights()
            assert w.dtype == np.float32 and np.array_equal(got, w), k
