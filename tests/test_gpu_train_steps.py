"""The two BF16 copies of the weights, one for the forward and one for the
backward pass, that a training step leaves to the next."""
import numpy as np
import pytest

from oracle import mlp
from gpu_common import vf  # noqa: F401
from test_gpu_nn import _gpu_training_set

pytestmark = pytest.mark.gpu

NAMES = ("W0", "b0", "W1", "b1", "W2", "b2", "W3", "b3")


def _layer(g, name):
    o, shp = mlp.blob_layout()[name]
    return g[o:o + int(np.prod(shp))]


@pytest.mark.parametrize("batch", [512, 1536])
def test_two_steps_are_adam_on_the_gradients(vf, batch):  # noqa: F811
    """Two steps against Adam in FP64 on vfisv_nn_grad at the weights before
    each.  A step's forward and backward pass read two BF16 copies of the
    weights, which the step before wrote and vfisv_nn_grad packs anew; a stale
    or misplaced element of either changes the second gradient.  All rows of
    the batch are one sample, so the order in which a step takes them changes
    no bit and the gradients are the same numbers: what is left are the
    roundings of the update in FP32, 2^-24 each: of the new weight; of the
    update's factors (lr, c1, c2 and v under the root, eps: five) and seven
    operations; and of m's two terms, which may cancel."""
    v, h, torch = vf
    tp, obs, _, _ = _gpu_training_set(v, h, torch, 4096, 71)
    blob0 = v.vfisv_nn_init(h, obs, tp, seed=9)
    obs, tp = (a[17:18].expand(batch, -1).contiguous() for a in (obs, tp))
    lr0 = float(np.float32(1e-2))
    one, two = blob0.clone(), blob0.clone()
    v.vfisv_nn_train(h, one, obs, tp, batch=batch, epochs=1, lr0=lr0, seed=5)
    hist = v.vfisv_nn_train(h, two, obs, tp, batch=batch, epochs=2, lr0=lr0, seed=5)
    (_, g1), (loss, g2) = (v.vfisv_nn_grad(h, b, obs, tp) for b in (blob0, one))
    v.vfisv_check(h)
    assert float(hist.reshape(-1)[1]) == float(loss.reshape(-1)[0])
    b1, b2 = float(np.float32(0.9)), float(np.float32(0.999))
    w = [b.double().cpu().numpy().reshape(-1)[:v.NN_NTRAIN] for b in (blob0, one, two)]
    g = [a.double().cpu().numpy().reshape(-1) for a in (g1, g2)]
    m = np.zeros_like(g[0])
    s = np.zeros_like(m)
    for t in (0, 1):
        lr = 0.5 * lr0 * (1.0 + np.cos(np.pi * t / 2.0))
        c1, c2 = 1.0 - b1 ** (t + 1), 1.0 - b2 ** (t + 1)
        mag = b1 * np.abs(m) + (1.0 - b1) * np.abs(g[t])
        m = b1 * m + (1.0 - b1) * g[t]
        s = b2 * s + (1.0 - b2) * g[t] ** 2
        f = lr / c1 / (np.sqrt(s / c2) + 1e-8)
        bound = 2.0 ** -24 * (np.abs(w[t + 1]) + 12.0 * f * np.abs(m) + f * mag) * 1.01
        err = np.abs(w[t + 1] - (w[t] - f * m))
        for name in NAMES:
            e, b = _layer(err, name), _layer(bound, name)
            assert np.all(e <= b), (t, name, float((e / b).max()))
