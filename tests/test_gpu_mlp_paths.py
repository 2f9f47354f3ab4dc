"""The two ways of training: up to 64 inputs and units in two launches an epoch, wider networks by
the general kernels with the epochs replayed from a captured graph.  Both give the gradient and
Adam calls' updates, and where a small network is widened by inputs and units that stay zero the
general kernels give its values bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _data(d, n, seed):
    rng = np.random.default_rng(seed)
    return rng.normal(0, 1, (n, d)).astype(np.float32), rng.normal(0, 1, n).astype(np.float32)


def _net(d, H, p):
    from paper_1204_4779_gb300 import costmodel
    net = costmodel.MLP(d, H, seed=1)
    net.set_params(p)
    return net


@pytest.mark.parametrize("d,H", [(10, 64), (70, 64), (20, 70)])
@pytest.mark.parametrize("epochs", [1, 15, 16, 17, 32, 37])
def test_training_equals_gradient_and_adam_steps(d, H, epochs):
    """16 epochs a graph: none, one or two replays and what is left over."""
    from paper_1204_4779_gb300 import costmodel
    X, t = _data(d, 300, 6)
    p = np.random.default_rng(7).normal(0, 0.4, costmodel.MLP(d, H).n_params)
    a, b = _net(d, H, p), _net(d, H, p)
    hist = a.train(X, t, epochs, lr=3e-3)
    losses = []
    for _ in range(epochs):
        g, loss = b.gradient(X, t)
        losses.append(loss)
        b.adam(g, lr=3e-3)
    # the same gradients and Adam formulas in two kernels, whose products the compiler may fuse
    # differently: an ulp or two of the update a step
    assert np.max(np.abs(a.get_params() - b.get_params())) <= 1e-5
    assert np.allclose(hist, losses, rtol=1e-5, atol=1e-7)


def _widen(p, d, H, D, G):
    """Flat parameters (W1, b1, W2, b2, W3, b3) of a d-H network as those of a D-G one, the added
    inputs and units zero; and the places of the original ones."""
    out, idx, o, q = np.zeros(G * D + G + G * G + G + G + 1, p.dtype), [], 0, 0
    for rows, cols, R, K in ((H, d, G, D), (H, 1, G, 1), (H, H, G, G), (H, 1, G, 1), (1, H, 1, G), (1, 1, 1, 1)):
        at = o + (np.arange(rows)[:, None] * K + np.arange(cols)[None, :]).ravel()
        out[at] = p[q:q + rows * cols]
        idx.append(at)
        o += R * K
        q += rows * cols
    return out, np.concatenate(idx)


@pytest.mark.parametrize("d,H,D,G", [(64, 64, 65, 64), (64, 64, 64, 65), (35, 17, 65, 65), (1, 1, 66, 70)])
@pytest.mark.parametrize("n", [1, 33, 130, 387])
def test_both_ways_give_the_same_bits(d, H, D, G, n):
    rng = np.random.default_rng(n + d)
    X, t = _data(d, n, n)
    XW = np.concatenate([X, np.zeros((n, D - d), np.float32)], 1)
    p = rng.normal(0, 0.3, H * d + H + H * H + H + H + 1).astype(np.float32)
    pw, idx = _widen(p, d, H, D, G)
    a, b = _net(d, H, p), _net(D, G, pw)
    ga, la = a.gradient(X, t)
    gb, lb = b.gradient(XW, t)
    assert la == lb and np.array_equal(ga, gb[idx])
    ha, hb = a.train(X, t, 20, lr=3e-3), b.train(XW, t, 20, lr=3e-3)
    assert np.array_equal(ha, hb) and np.array_equal(a.get_params(), b.get_params()[idx])
