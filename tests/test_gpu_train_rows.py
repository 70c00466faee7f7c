"""What the training step's kernels may not lose between them: a row of the
batch on its way into the gradients' sums."""
import numpy as np
import pytest

from oracle import mlp
from gpu_common import f32, vf  # noqa: F401
from test_gpu_nn import _oracle_set, _random_blob

pytestmark = pytest.mark.gpu

NAMES = ("W0", "b0", "W1", "b1", "W2", "b2", "W3", "b3")


def _layer(g, name):
    o, shp = mlp.blob_layout()[name]
    return np.asarray(g, np.float64).reshape(-1)[o:o + int(np.prod(shp))]


@pytest.mark.parametrize("n", [65, 129, 300, 2049])
def test_every_row_counts_once(vf, n):  # noqa: F811
    """A row of every 64-row chunk, the first and the last among them, in turn
    gets a target (B, far from the others') that makes it the better part of
    the gradient: in the oracle, leaving such a row out changes every layer's
    gradient by 78 % or more in these sizes.  Bound on the relative L2 error
    against the oracle's rounded-operand reading as in the tests of the tile
    edges: a step of 2^-8 for each operand of the four products behind it."""
    v, h, torch = vf
    p, obs, _ = _oracle_set(n, 61 + n)
    p0, obs0, _ = _oracle_set(400, 7)
    blob = _random_blob(3, obs0, p0)
    far = 1e3 * np.sqrt(n) * np.ravel(mlp.unpack(blob)[1]["out_std"])[0]
    chunks = [64 * c + 11 * c % 64 for c in range(n // 64)]
    for r in sorted({0, n - 1, *chunks}):
        q = p.copy()
        q[r, 0] = f32(q[r, 0] + far)
        L_b, g_b, _ = mlp.loss_and_grad(blob, obs, q, operand_round=mlp.round_bf16)
        loss, g = v.vfisv_nn_grad(h, blob.astype(np.float32), obs.astype(np.float32),
                                  q.astype(np.float32))
        for name in NAMES:
            a, b = _layer(g, name), _layer(g_b, name)
            rel = np.linalg.norm(a - b) / np.linalg.norm(b)
            assert rel < 4 * 2.0 ** -8, (r, name, rel)
        assert abs(loss[0] / L_b - 1) < 1e-3, r
    v.vfisv_check(h)
