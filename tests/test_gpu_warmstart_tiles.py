"""The warm-start convolutions at the edges of their 16 x 16 tiles and of their work split, and
the minibatches of lb_ws_train, against the numpy oracle.

Tolerances: a float32 sum of K = 288 products is off by at most K 2^-24 = 1.7e-5 of the sum of
their magnitudes.  A forward pass chains four such layers (7e-5 of the largest output); a gradient
chains up to eight and a sum over pixels (4e-4 of its norm)."""
import numpy as np
import pytest

from oracle import cnn_oracle as C
from tests.helpers import library
from tests.test_gpu_warmstart_net import CHANNELS, _as_fp16_params, _packed, _unpack

pytestmark = pytest.mark.gpu


def _net(seed):
    rng = np.random.default_rng(seed)
    return [(W, rng.uniform(-0.1, 0.1, b.shape)) for W, b in C.init_params(CHANNELS, seed=seed)], rng


# one pixel, one tile, a row or a column more, widths that are and are not a multiple of four, and
# more tiles than CTAs of the weight-gradient kernel
@pytest.mark.parametrize("n,H,W", [(1, 1, 1), (2, 16, 16), (1, 17, 20), (1, 3, 18), (2, 15, 33), (1, 40, 8), (20, 64, 68)])
def test_layers(n, H, W):
    lb = library()
    params, rng = _net(11)
    x = rng.uniform(-1, 1, (n, 5, H, W)).astype(np.float32)
    t = rng.uniform(-1, 1, (n, 3, H, W)).astype(np.float32)
    with lb.WarmStart() as ws:
        ws.set_params(_packed(params))
        y = ws.forward(x)
        loss, g = ws.loss_grad(x, t)
    p16 = _as_fp16_params(params)
    want, _ = C.forward(x.astype(np.float64), p16)
    assert np.abs(y - want).max() <= 7e-5 * np.abs(want).max()
    want_loss, grads = C.loss_and_grads(x.astype(np.float64), t.astype(np.float64), p16)
    assert abs(loss - want_loss) <= 4e-4 * want_loss
    for (dW, db), (wW, wb) in zip(_unpack(g.astype(np.float64), params), grads):
        assert np.linalg.norm(dW - wW) <= 4e-4 * np.linalg.norm(wW)
        assert np.linalg.norm(db - wb) <= 4e-4 * np.linalg.norm(wb)


def test_minibatches():
    """Seven samples in minibatches of three for two epochs: the shuffled order, the sample that is
    left out, Adam and the loss of each epoch.  The first steps of Adam move every weight by about
    the learning rate whatever its gradient's size, so a wrong sample shows at once."""
    lb = library()
    params, rng = _net(12)
    n, batch, epochs, lr, seed = 7, 3, 2, 1e-3, 5
    x = rng.uniform(-1, 1, (n, 5, 9, 14)).astype(np.float32)
    t = rng.uniform(-1, 1, (n, 3, 9, 14)).astype(np.float32)
    p0 = _packed(params)
    with lb.WarmStart() as ws:
        ws.set_params(p0)
        hist = ws.train(x, t, epochs=epochs, batch=batch, lr=lr, seed=seed)
        got = ws.get_params()
    mask = (1 << 64) - 1
    rs = (seed * 0x9E3779B97F4A7C15 + 1) & mask
    order, p = list(range(n)), p0.astype(np.float64)
    m, v, k = np.zeros_like(p), np.zeros_like(p), 0
    for e in range(epochs):
        for i in range(n - 1, 0, -1):
            rs ^= (rs << 13) & mask
            rs ^= rs >> 7
            rs ^= (rs << 17) & mask
            j = rs % (i + 1)
            order[i], order[j] = order[j], order[i]
        losses = []
        for b in range(n // batch):
            pick = order[b * batch:(b + 1) * batch]
            loss, grads = C.loss_and_grads(x[pick].astype(np.float64), t[pick].astype(np.float64),
                                           _as_fp16_params(_unpack(p, params)))
            g = np.concatenate([np.concatenate([dW.reshape(-1), db]) for dW, db in grads])
            k += 1
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            p = p - lr * (m / (1 - 0.9 ** k)) / (np.sqrt(v / (1 - 0.999 ** k)) + 1e-8)
            losses.append(loss)
        assert abs(hist[e] - np.mean(losses)) <= 4e-4 * np.mean(losses)
    assert np.linalg.norm(got - p) <= 1e-2 * np.linalg.norm(p - p0)
