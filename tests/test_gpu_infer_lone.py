"""Inference up to one 128-pixel tile an SM, where all compute warps share a
CTA's one tile, against calls with more tiles, where they form two groups: a
pixel's outputs are the same bits."""
import numpy as np
import pytest

from gpu_common import LINE, vf  # noqa: F401
from test_gpu_nn import _gpu_training_set

pytestmark = pytest.mark.gpu


def test_one_tile_and_more(vf):  # noqa: F811
    v, h, torch = vf
    full = torch.cuda.get_device_properties(0).multi_processor_count * 128
    tp, obs, _, _ = _gpu_training_set(v, h, torch, full + 1, 91)
    blob = v.vfisv_nn_init(h, obs, tp, seed=9)
    more = v.vfisv_nn_infer(h, blob, obs, LINE, want_raw=True)  # one CTA has two tiles
    for n in (1, 127, 128, 129, full - 1, full):
        one = v.vfisv_nn_infer(h, blob, obs[:n].contiguous(), LINE, want_raw=True)
        for key in ("init", "conf", "raw"):
            x, y = (a.cpu().numpy().view(np.int32) for a in (more[key][:n], one[key]))
            assert np.array_equal(x, y), (n, key)
    v.vfisv_check(h)
