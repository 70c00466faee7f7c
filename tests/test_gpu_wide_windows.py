"""The wide kernels' two ways of applying the instrument profiles and their
edges: regular bands (windows of up to eight groups of four points, samples
whose bands the grid cuts off at its ends, grids that end inside a chunk of 64
or a group of 4), irregular ones (unevenly spaced samples, a profile wider
than the others' windows allow), a sample without transmission.  Synthesis and
the fit's starting chi2 (iteration cap 0, at the true model and at another)
against the oracle: Stokes within the synthesis bound of 1e-5 I_c, and chi2
within the size that bound gives it: with residuals r and weights w, d chi2 <=
sum(2 w |r| 1e-5 + w 1e-10) / dof."""
import numpy as np
import pytest

import workloads as W
from oracle import me
from gpu_common import f32, vf  # noqa: F401

pytestmark = pytest.mark.gpu
LINE = W.FE6302


def _instrument(kind):
    if kind == "regular":  # 16 samples, 4 points apart, cut off at both ends
        x, c = W.spectrograph_grid(16, 21.5, 4)
        return W.spectrograph_instrument(x, c), x
    if kind == "ragged":  # the grid ends inside a group and a chunk
        x, c = W.spectrograph_grid(19, 21.5, 4)
        T = W.spectrograph_instrument(x, c)[:, :75]
        T[:, 70:] *= 0.5
        return T[:18], x[:75]
    if kind == "wide":  # eight groups a window
        x, c = W.spectrograph_grid(40, 21.5, 4)
        return W.spectrograph_instrument(x, c, fwhm_mA=27.5), x
    if kind == "uneven":
        x, _ = W.spectrograph_grid(30, 21.5, 4)
        c = x[0] + (x[-1] - x[0]) * np.linspace(0.1, 0.9, 20) ** 1.7
        return W.spectrograph_instrument(x, c), x
    x, c = W.spectrograph_grid(33, 21.5, 4)  # "dark": one sample sees nothing
    T = W.spectrograph_instrument(x, c)
    T[11] = 0.0
    return T, x


@pytest.mark.parametrize("kind", ["regular", "ragged", "wide", "uneven", "dark"])
def test_profiles_and_edges(vf, kind):
    v, h, torch = vf
    T, x = (f32(a) for a in _instrument(kind))
    nf, n = T.shape[0], 60
    p = f32(W.quiet_and_active_params(n, 17))
    ps = p.copy()
    ps[::4, 9] = 0.6
    ps = f32(ps)
    s = v.vfisv_synth(h, ps.astype(np.float32), T.astype(np.float32), x.astype(np.float32), LINE)
    assert np.abs(s - me.synth(ps, T, x, LINE)).max() <= 1e-5
    syn = me.synth(p, T, x, LINE).reshape(n, -1)
    obs = f32(syn + 1e-3 * W.noise(n, 4 * nf, 17))
    w = f32(np.full(4 * nf, 1e6))
    other = p.copy()
    other[:, 0] *= 1.1
    for m in (p, f32(other)):
        r = v.vfisv_invert(h, obs.astype(np.float32), w.astype(np.float32), T.astype(np.float32),
                           x.astype(np.float32), LINE, init=m.astype(np.float32),
                           config={"max_iter": 0})
        v.vfisv_check(h)
        res = obs - me.synth(m, T, x, LINE).reshape(n, -1)
        dof = 4 * nf - 9
        ref = (w * res * res).sum(1) / dof
        tol = (2e-5 * w * np.abs(res) + w * 1e-10).sum(1) / dof
        assert (np.abs(r["chi2"] - ref) <= tol + 1e-6 * ref).all()
