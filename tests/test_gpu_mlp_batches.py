"""Training gradients over batches of every tiling: part of a 32-row tile, a
whole number of tiles, one and several tiles per block."""
import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rb():
    from paper_1110_4876_gb300 import build, rb as _rb
    build.build()
    _rb.load()
    return _rb


@pytest.mark.parametrize("n", [1, 15, 16, 17, 31, 32, 33, 64, 2047, 152 * 32, 152 * 32 + 1, 10_007])
def test_gradient_matches_oracle(rb, n):
    """BF16 operands (relative rounding 2^-9 each, three products deep) with
    FP32 sums: every layer's gradient within 1e-2 in norm of the FP64 backward
    pass, 2e-2 below 64 rows, where fewer roundings average out."""
    g = np.random.default_rng(n)
    theta = omlp.init(3)
    X = g.normal(0, 1, (n, 12))
    Y = g.normal(0, 0.3, (n, 3))
    L_ref, ref = omlp.backward(theta, X, Y)
    grad, L = rb.rb_mlp_grad(theta, X, Y)
    tol = 1e-2 if n >= 64 else 2e-2
    assert L == pytest.approx(L_ref, rel=tol)
    k = 0
    for a, b in zip(omlp.SIZES[:-1], omlp.SIZES[1:]):
        for size in (a * b, b):
            d = np.linalg.norm(grad[k: k + size] - ref[k: k + size])
            assert d <= tol * np.linalg.norm(ref[k: k + size]) + 1e-12, (k, size)
            k += size


def test_gradient_is_the_same_on_every_run(rb):
    """Sums run in a fixed order."""
    g = np.random.default_rng(1)
    theta, X, Y = omlp.init(4), g.normal(0, 1, (5001, 12)), g.normal(0, 0.3, (5001, 3))
    a, la = rb.rb_mlp_grad(theta, X, Y)
    b, lb = rb.rb_mlp_grad(theta, X, Y)
    assert np.array_equal(a, b) and la == lb


@pytest.mark.parametrize("n", [16, 100, 152 * 32 + 2])
def test_training_is_adam_on_the_gradients(rb, n):
    """One batch per epoch of columns of +-1 (mean 0 and variance 1, so
    standardising changes nothing): the weights after three epochs are three
    Adam steps on the gradients.  A step moves a weight by lr m / sqrt(v); a
    gradient may differ by 2^-8 where a weight rounds to the other BF16 value,
    so steps agree to 3 x 2^-8 of lr each, doubled; weights whose gradients are
    below 1e-5 are left out (rounding of the sums, 1e-7 of the terms, next to
    Adam's 1e-8)."""
    g = np.random.default_rng(n)
    theta = omlp.init(5)
    X = g.choice([-1.0, 1.0], (n, 12))
    Y = g.choice([-1.0, 1.0], (n, 3))
    X[1::2], Y[1::2] = -X[0::2], -Y[0::2]
    lr = 1e-3
    w, _ = rb.rb_mlp_train(X, Y, theta, epochs=3, batch=n, lr=lr, seed=1)
    ref = theta.astype(np.float32).astype(np.float64)
    m, v = np.zeros_like(ref), np.zeros_like(ref)
    keep = np.ones(len(ref), bool)
    for step in range(1, 4):
        grad, _ = rb.rb_mlp_grad(ref, X, Y)
        keep &= np.abs(grad) > 1e-5
        m = 0.9 * m + 0.1 * grad
        v = 0.999 * v + 0.001 * grad.astype(np.float64) ** 2
        ref = ref - lr * (m / (1 - 0.9**step)) / (np.sqrt(v / (1 - 0.999**step)) + 1e-8)
    assert keep.mean() > 0.9
    assert np.abs(w - ref)[keep].max() <= 2 * 3 * 3 * 2.0**-8 * lr
