"""What an inversion without a set launch shape may not depend on: the kernel
that the size of the map selects."""
import numpy as np
import pytest

import workloads as W
from gpu_common import LINE, vf  # noqa: F401

pytestmark = pytest.mark.gpu


def _map(v, h, torch, n, x, seed=5):
    t = lambda a: torch.tensor(np.asarray(a, np.float32), device="cuda:0")  # noqa: E731
    p = W.quiet_and_active_params(n, seed)
    tf, tx = t(W.hmi_filters(x)), t(x)
    syn = v.vfisv_synth(h, t(p), tf, tx, LINE).reshape(n, 24)
    sig = 1e-3 * t(W.continuum(p))[:, None]
    obs = (syn + sig * t(W.noise(n, 24, seed))).contiguous()
    return obs, (1.0 / (sig * sig)).expand(n, 24).contiguous(), tf, tx


@pytest.mark.parametrize("nlam,big,small", [(297, 263, 200), (297, 200, 100), (450, 394, 200),
                                            (149, 300, 80), (2000, 300, 200)])
def test_a_smaller_map_needs_no_larger_workspace(vf, nlam, big, small):  # noqa: F811
    """A call under capture may not grow the workspace: after an uncaptured call
    on a map, any smaller one on the same grid is captured, whichever kernels
    the two take (sizes in pixels an SM)."""
    v, _, torch = vf
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    h = v.vfisv_create(0)
    obs, w, tf, tx = _map(v, h, torch, big * sms, np.linspace(-740.0, 740.0, nlam))
    n = small * sms
    cfg = {"max_iter": 2}
    s = torch.cuda.Stream(torch.device("cuda:0"))
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        ref = v.vfisv_invert(h, obs, w, tf, tx, LINE, config=cfg, stream=s)
        s.synchronize()
        out = {k: torch.empty_like(r[:n]) for k, r in ref.items()}
        v.vfisv_graph_begin(h, s)
        v.vfisv_invert(h, obs[:n], w[:n], tf, tx, LINE, config=cfg, out=out, stream=s)
        g = v.vfisv_graph_end(h, s)
        g.launch(s)
        s.synchronize()
    for k in out:
        assert torch.equal(out[k], ref[k][:n]), k
    v.vfisv_check(h)
    g.close()
    h.close()
