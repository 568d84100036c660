"""The training kernel where its split changes: minibatches of one tile, of two (up
to 256 samples), of several passes with a remainder, and features that do not start
at 16 bytes.

Bounds, from the arithmetic: a gradient is a sum of fp32 products in a fixed order,
off by up to 1e-5 of the sum of its terms' magnitudes, 1e-3 of itself where the
terms cancel a hundredfold, and one sample's unit on the other side of zero moves
it by at most a two-hundredth; Adam turns that share of a gradient into the same
share of a step, lr = 0.01.  At most 12 steps: 2e-4 (and 2e-3 of a weight), as
where whole training runs are compared.  A tile that is left out or counted twice
moves weights by steps of 0.01 and the losses by percents.
"""
import ctypes

import numpy as np
import pytest

from oracle import mlp
from paper_1709_09990_gb300 import graphgen as gg
from tests.gpu_util import context

pytestmark = pytest.mark.gpu


def _case(B, epochs, seed):
    rng = np.random.default_rng(seed)
    x = rng.random((B, 12)).astype(np.float32)
    y = (x[:, :3].sum(axis=1) / 3).astype(np.float32)
    r = gg.Rng(seed)
    p = np.array([(r.uniform() - 0.5) * 0.6 for _ in range(mlp.N_PARAMS)], dtype=np.float32)
    return x, y, p, np.stack([rng.permutation(B) for _ in range(epochs)]).astype(np.int32)


def _reference(x, y, p0, perm, minibatch):
    p, losses, t = p0.astype(np.float64), [], 0
    m, v = np.zeros_like(p), np.zeros_like(p)
    for order in perm:
        total = 0.0
        for s in range(0, len(order), minibatch):
            idx = order[s: s + minibatch]
            _, _, yh = mlp.forward(p, x[idx])
            total += float(((yh - y[idx]) ** 2).sum())
            t += 1
            p, m, v = mlp.adam_step(p, mlp.grad(p, x[idx], y[idx]), m, v, t, lr=0.01)
        losses.append(total / len(order))
    return p, losses


@pytest.mark.parametrize("B,minibatch", [(1, 1), (127, 200), (256, 128), (400, 129), (600, 200), (700, 256), (512, 255),
                                         (900, 300), (700, 700), (1500, 513)])
def test_minibatches_across_tiles_and_passes(B, minibatch):
    x, y, p0, perm = _case(B, 2, B + minibatch)
    p = p0.copy()
    with context() as c:
        loss = c.mlp_train(p, x, y, minibatch, perm, lr=0.01)
    ref, losses = _reference(x, y, p0, perm, minibatch)
    np.testing.assert_allclose(p, ref, rtol=2e-3, atol=2e-4)
    np.testing.assert_allclose(loss, losses, rtol=1e-3)


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
def test_features_anywhere_on_the_device(shift):
    torch = pytest.importorskip("torch")
    from paper_1709_09990_gb300 import native
    B, minibatch, epochs = 500, 300, 2
    x, y, p0, perm = _case(B, epochs, 77)
    buf = torch.zeros(B * 12 + 4, dtype=torch.float32, device="cuda")
    buf[shift: shift + B * 12] = torch.from_numpy(x.reshape(-1)).cuda()
    torch.cuda.synchronize()
    p, loss = p0.copy(), np.zeros(epochs, np.float32)
    with context() as c:
        rc = native.lib().tw_mlp_train(c._h, p.ctypes.data, buf.data_ptr() + 4 * shift, y.ctypes.data, B, minibatch,
                                       epochs, perm.ctypes.data, ctypes.c_float(0.01), loss.ctypes.data)
        assert rc == native.TW_OK
        again = p0.copy()
        loss2 = c.mlp_train(again, x, y, minibatch, perm, lr=0.01)
    # the same sums in the same order, wherever the features lie
    assert np.array_equal(p, again) and np.array_equal(loss, loss2)
    ref, losses = _reference(x, y, p0, perm, minibatch)
    np.testing.assert_allclose(p, ref, rtol=2e-3, atol=2e-4)
    np.testing.assert_allclose(loss, losses, rtol=1e-3)
