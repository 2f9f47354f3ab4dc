"""Gradients and training of small networks at the edges of the two-launch epoch's tiles (32
samples), chunks (128 samples, a cluster each) and units per CTA (16), and at the line to the
general kernels (64 inputs, 64 units), against the FP64 CPU oracle."""
import numpy as np
import pytest

from oracle import mlp_oracle as M

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("d,H", [(1, 1), (7, 17), (35, 64), (64, 64), (65, 64), (64, 65)])
@pytest.mark.parametrize("n", [1, 31, 33, 128, 130, 387])
def test_gradient_matches_oracle(d, H, n):
    from paper_1204_4779_gb300 import costmodel
    rng = np.random.default_rng(1000 * d + 10 * H + n)
    net = costmodel.MLP(d, H, seed=1)
    p = rng.normal(0, 0.3, net.n_params).astype(np.float32)
    net.set_params(p)
    X = rng.normal(0, 1, (n, d)).astype(np.float32)
    t = rng.normal(0, 1, n).astype(np.float32)
    g, loss = net.gradient(X, t)
    q, Xd, td = p.astype(np.float64), X.astype(np.float64), t.astype(np.float64)
    go, lo = M.gradient(q, Xd, td, d, H), M.loss(q, Xd, td, d, H)
    # sums of up to ~130 FP32 terms per sample and layer: a few hundred roundings of 6e-8
    assert abs(loss - lo) <= 3e-5 * max(1.0, lo)
    assert np.max(np.abs(g - go)) <= 1e-4 * max(1e-3, np.max(np.abs(go)))
    a = net.train(X, t, 3, lr=1e-3)
    assert abs(a[0] - loss) == 0.0 and np.all(np.isfinite(a))
