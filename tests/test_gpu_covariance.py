"""The covariance's paths for numerically singular pixels: the eigen fallback
runs one pixel a lane where a CTA has warps full of them and by groups of
lanes for the few left over.  Each row depends on its pixel alone, so the same
pixels called in maps of other sizes (other CTAs, other queues, other paths)
give the same rows bit for bit; quiet pixels with next to no field leave B,
gamma and psi undetermined, so many of them are singular."""
import numpy as np
import pytest

import workloads as W
from gpu_common import LINE, T, X, vf  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mask,fast", [(0x1FF, 0), (0x1FF, 1), (0x3FF, 0), (0x1F7, 0)])
def test_rows_do_not_depend_on_the_map(vf, mask, fast):
    v, h, torch = vf
    n = 12000
    dev = torch.device("cuda:0")
    t = lambda a: torch.tensor(np.asarray(a, np.float32), device=dev)  # noqa: E731
    p = W.quiet_and_active_params(n, 77, b_max=1e-3)
    p[::2, 0] *= 1e5
    tf, tx = t(T), t(X)
    obs = v.vfisv_synth(h, t(p), tf, tx, LINE).reshape(n, 24) + 1e-3 * t(W.noise(n, 24, 77))
    w = torch.full((24,), 1e6, device=dev)
    init = t(p)
    cfg = {"max_iter": 0, "free_mask": mask, "fast_solve": fast}
    full = v.vfisv_invert(h, obs, w, tf, tx, LINE, init=init, config=cfg)["cov"]
    full = full.view(torch.int32)  # bits: some variances leave FP32's range
    assert (full != 0).any()
    for a, b in ((0, 1), (5, 38), (100, 1100), (3000, 8000), (11999, 12000)):
        part = v.vfisv_invert(h, obs[a:b].contiguous(), w, tf, tx, LINE,
                              init=init[a:b].contiguous(), config=cfg)["cov"]
        assert torch.equal(full[a:b], part.view(torch.int32)), (a, b)
    v.vfisv_check(h)
