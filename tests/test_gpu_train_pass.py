"""The training step's kernels at the edges of their tiles: batches around one
128-row tile and one 64-row K-chunk of the weight gradients, and the weights
that a step hands to the next."""
import numpy as np
import pytest

from oracle import mlp
from gpu_common import vf  # noqa: F401
from test_gpu_nn import _gpu_training_set, _oracle_set, _random_blob

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 63, 65, 128, 129, 300, 2049])
def test_gradient_tile_edges(vf, n):  # noqa: F811
    """Each layer's gradient in relative L2 against the oracle's rounded-operand
    reading.  The two differ where an FP32 sum lands on the other side of a
    bfloat16 rounding; were that so for every operand of the four products
    behind a gradient, each would add one step of 2^-8, so 4 * 2^-8 bounds it
    for any n (a lost or doubled row is far above it in these sizes)."""
    v, h, torch = vf
    p, obs, w = _oracle_set(n, 61 + n)
    p0, obs0, _ = _oracle_set(400, 7)
    blob = _random_blob(3, obs0, p0)
    L_b, g_b, _ = mlp.loss_and_grad(blob, obs, p, operand_round=mlp.round_bf16)
    loss, g = v.vfisv_nn_grad(h, blob.astype(np.float32), obs.astype(np.float32),
                              p.astype(np.float32))
    v.vfisv_check(h)
    lay = mlp.blob_layout()
    for name in ("W0", "b0", "W1", "b1", "W2", "b2", "W3", "b3"):
        o, shp = lay[name]
        e = int(np.prod(shp))
        a, b = g[o:o + e].astype(np.float64), g_b[o:o + e]
        rel = np.linalg.norm(a - b) / np.linalg.norm(b)
        print(f"n {n} {name}: {rel:.2e}")
        assert rel < 4 * 2.0 ** -8, (name, rel)
    assert abs(loss[0] / L_b - 1) < 1e-3


@pytest.mark.parametrize("batch", [512, 1536, 4608])
def test_step_hands_its_weights_on(vf, batch):  # noqa: F811
    """With one batch an epoch, the second step's loss is the loss of the
    weights after the first: the same rows in another order, so the two differ
    by the order of an FP32 sum of `batch` positive terms alone."""
    v, h, torch = vf
    tp, obs, tf, tx = _gpu_training_set(v, h, torch, batch, 71)
    blob0 = v.vfisv_nn_init(h, obs, tp, seed=9)
    one = blob0.clone() if torch.is_tensor(blob0) else blob0.copy()
    two = blob0.clone() if torch.is_tensor(blob0) else blob0.copy()
    v.vfisv_nn_train(h, one, obs, tp, batch=batch, epochs=1, lr0=1e-3, seed=5)
    hist = v.vfisv_nn_train(h, two, obs, tp, batch=batch, epochs=2, lr0=1e-3, seed=5)
    loss, _ = v.vfisv_nn_grad(h, one, obs, tp)
    v.vfisv_check(h)
    want = float(loss.reshape(-1)[0])
    assert abs(float(hist.reshape(-1)[1]) / want - 1) < batch * 2.0 ** -23
