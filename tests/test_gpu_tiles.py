"""Edges of the tiled preparation kernels, of the packed synthesis loop and of
the filter-table packing.

* The weights and the weak-field models depend on their pixel alone, so a
  call on the pixels from `off` on gives the rows of the whole call bit for
  bit, whatever tile and alignment a pixel falls on.
* Synthesis takes two grid points a round: grids with an odd and an even
  number of kept points, one point, and tables past the packing's
  shared-memory copy, against the oracle within the synthesis bound (1e-5 of
  the continuum)."""
import numpy as np
import pytest

import workloads as W
from oracle import me
from gpu_common import LINE, T, X, f32, vf  # noqa: F401

pytestmark = pytest.mark.gpu


def _unaligned(torch, a):
    """The same values at an address 4 bytes past a 16-byte boundary."""
    buf = torch.empty(a.numel() + 1, dtype=a.dtype, device=a.device)
    buf[1:] = a.reshape(-1)
    return buf[1:].view(a.shape)


@pytest.mark.parametrize("nf", [3, 6, 8])
@pytest.mark.parametrize("n,off", [(2, 1), (129, 1), (300, 127), (513, 256)])
def test_preparation_tiles(vf, n, off, nf):
    v, h, torch = vf
    dev = torch.device("cuda:0")
    c = (np.arange(nf) - (nf - 1) / 2.0) * 69.0
    t = lambda a: torch.tensor(np.asarray(a, np.float32), device=dev)  # noqa: E731
    tf, tx = t(W.hmi_filters(X, centres_mA=c)), t(X)
    p = t(W.quiet_and_active_params(n, 31))
    obs = v.vfisv_synth(h, p, tf, tx, LINE).reshape(n, 4 * nf)
    obs = obs + 1e-3 * t(W.noise(n, 4 * nf, 31))
    if n > 200:
        obs[5, 1] = float("nan")
    mu = torch.linspace(0.1, 1.0, n, device=dev)
    full = v.vfisv_init_models(h, obs, tf, tx, LINE)
    w = v.vfisv_limb_weights(h, obs, mu, 1.0, [1e-3, 2e-3, 2e-3, 1e-3])
    for o in (obs[off:], _unaligned(torch, obs[off:])):
        part = v.vfisv_init_models(h, o, tf, tx, LINE)
        for k in ("init", "pol"):
            assert torch.equal(torch.nan_to_num(full[k][off:], nan=-9.0),
                               torch.nan_to_num(part[k], nan=-9.0)), k
        wp = v.vfisv_limb_weights(h, o, mu[off:].contiguous(), 1.0, [1e-3, 2e-3, 2e-3, 1e-3])
        assert torch.equal(torch.nan_to_num(w[off:], nan=-9.0), torch.nan_to_num(wp, nan=-9.0))


@pytest.mark.parametrize("nlam,nf", [(1, 1), (2, 6), (3, 6), (62, 1), (63, 8), (1024, 8), (1025, 6)])
def test_synthesis_point_pairs(vf, nlam, nf):
    v, h, torch = vf
    x = W.wavelength_grid(nlam, 1480.0 / max(nlam, 2))
    c = (np.arange(nf) - (nf - 1) / 2.0) * 69.0
    Tn = W.hmi_filters(x, centres_mA=c)
    p = W.quiet_and_active_params(130, 7)
    p[::3, 9] = 0.4
    s = v.vfisv_synth(h, p.astype(np.float32), Tn.astype(np.float32), x.astype(np.float32), LINE)
    ref = me.synth(f32(p), f32(Tn), f32(x), LINE)
    assert np.abs(s - ref).max() <= 1e-5
