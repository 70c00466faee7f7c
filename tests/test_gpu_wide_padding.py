"""Points of the fine grid that no sample sees (zero in every profile) take no
part in a spectrograph fit, whatever their wavelength says: a grid padded at
its end with NaN or far-off values fits like the grid without the padding, bit
for bit (the pixels' chunks of 64 points start at the same places)."""
import numpy as np
import pytest

import workloads as W
from gpu_common import vf  # noqa: F401

pytestmark = pytest.mark.gpu
LINE = W.FE6302


@pytest.mark.parametrize("fwhm", [10.0, 17.0, 25.0])
@pytest.mark.parametrize("pad", [np.nan, np.inf, 1e30, 0.0])
@pytest.mark.parametrize("extra", [3, 12, 40])
def test_padding_of_the_grid(vf, fwhm, pad, extra):  # noqa: F811
    v, h, torch = vf
    t = lambda a: torch.tensor(np.asarray(a, np.float32), device="cuda:0")  # noqa: E731
    x, c = W.spectrograph_grid(40, 21.5, 4)
    T = W.spectrograph_instrument(x, c, fwhm_mA=fwhm)
    n = 40
    p = t(W.quiet_and_active_params(n, 23))
    obs = v.vfisv_synth(h, p, t(T), t(x), LINE).reshape(n, -1)
    obs = (obs + 1e-3 * t(W.noise(n, 160, 23))).contiguous()
    w = torch.full((160,), 1e6, device="cuda:0")
    cfg = {"max_iter": 12}
    a = v.vfisv_invert(h, obs, w, t(T), t(x), LINE, config=cfg)
    v.vfisv_check(h)
    Tp = np.concatenate([T, np.zeros((40, extra))], axis=1)
    xp = np.concatenate([x, np.full(extra, pad)])
    b = v.vfisv_invert(h, obs, w, t(Tp), t(xp), LINE, config=cfg)
    v.vfisv_check(h)
    assert bool((a["status"] <= 2).all())
    for k in a:
        assert torch.equal(a[k], b[k]), k
