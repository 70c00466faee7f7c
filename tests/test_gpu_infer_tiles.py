"""Inference with one, two and an odd number of 128-pixel tiles a CTA: a pixel's
outputs do not depend on the tile that it falls in, so a call's outputs are bit
for bit those of its parts."""
import numpy as np
import pytest

from gpu_common import LINE, vf  # noqa: F401
from test_gpu_nn import _gpu_training_set

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tiles,rest", [(1, 1), (2, -1), (3, 5), (5, -127)])
def test_infer_parts(vf, tiles, rest):  # noqa: F811
    v, h, torch = vf
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = tiles * sms * 128 + rest
    tp, obs, _, _ = _gpu_training_set(v, h, torch, n, 81 + tiles)
    blob = v.vfisv_nn_init(h, obs, tp, seed=9)
    whole = v.vfisv_nn_infer(h, blob, obs, LINE, want_raw=True)
    v.vfisv_check(h)
    part = 61 * 128 + 37  # no multiple of a tile, less than one tile an SM
    for a in list(range(0, n, 9 * part))[:6] + [n - part]:
        one = v.vfisv_nn_infer(h, blob, obs[a:a + part].contiguous(), LINE, want_raw=True)
        for key in ("init", "conf", "raw"):
            x, y = whole[key][a:a + part], one[key]
            assert np.array_equal(x.cpu().numpy().view(np.int32), y.cpu().numpy().view(np.int32)), key
