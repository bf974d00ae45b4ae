"""The estimator's gradient over batches around the kernel's edges: tiles of
32 samples, blocks of at least 21, at most 304 blocks.  The inputs make the
forward pass exact in FP32 (small multiples of 1/4), so no ReLU or loss
branch can fall the other way, and the gradients are held to the rounding
bound of their sums: a 64-term dot product, then a block's samples one after
the other and the blocks' shares."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

I, H = 16, 64


@pytest.fixture(scope="module")
def cdl():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a GPU"
    from paper_2501_13051_gb300 import build as B
    B.build()
    from paper_2501_13051_gb300 import cdl as C
    return C


@pytest.mark.parametrize("n", [1, 7, 20, 21, 22, 31, 32, 33, 41, 42, 43, 672, 6383, 6384, 6385, 20001])
def test_gradient_of_a_batch(cdl, n):
    import torch
    rng = np.random.default_rng(n)
    q = lambda *s: rng.integers(-2, 3, s) / 4.0
    w1, b1, w2, b2, w3, b3 = q(H, I), q(H), q(H, H), q(H), q(H), q(1)
    X, y = rng.integers(0, 4, (n, I)).astype(np.float64), rng.integers(-40, 40, n) / 2.0
    th = np.concatenate([a.ravel() for a in (w1, b1, w2, b2, w3, b3)])
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    tau = 0.75
    pred, grad = cdl.mlp_gradient(f(th), f(X), f(y), tau=tau)
    fwd = cdl.mlp_forward(f(th), f(X))

    h1 = np.maximum(X @ w1.T + b1, 0)
    h2 = np.maximum(h1 @ w2.T + b2, 0)
    p = h2 @ w3 + b3[0]
    assert np.array_equal(pred.cpu().numpy(), p.astype(np.float32))
    assert np.array_equal(fwd.cpu().numpy(), p.astype(np.float32))

    def grads(g, w2, w3):
        g2 = g[:, None] * w3 * (h2 > 0)
        g1 = (g2 @ w2) * (h1 > 0)
        return np.concatenate([(g1.T @ X).ravel(), g1.sum(0), (g2.T @ h1).ravel(), g2.sum(0), g @ h2,
                               [g.sum()]])

    g = np.where(y > p, -tau, 1 - tau) / n
    want, size = grads(g, w2, w3), grads(np.abs(g), np.abs(w2), np.abs(w3))
    blocks = min(max(n // 21, 1), 304)
    terms = H + 4 + (n + blocks - 1) // blocks + (blocks + 7) // 8 + 8
    assert np.all(np.abs(grad.cpu().numpy() - want) <= terms * 2.0 ** -24 * size)
