"""The warp-specialised LM kernel's batches of pixel slots against 128 x 1, bit
for bit: a map larger than the 384 slots an SM holds, so that slots refill from
the queue, and the two batches a sub-partition that filter tables of more than
1,584 points leave room for, with one and both of them in flight and refilling
(maps of so many pixels an SM; one SM's 128 slots are a batch)."""
import numpy as np
import pytest

import workloads as W
from gpu_common import LINE, vf  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nlam,sms,per_sm", [
    (149, 0, 461), (1584, 5, 300), (1584, 5, 420), (1585, 5, 128), (1585, 5, 129),
    (1585, 5, 256), (1585, 5, 333), (4096, 5, 200), (4096, 5, 301)])
def test_same_bits(vf, nlam, sms, per_sm):  # noqa: F811
    v, _, torch = vf
    t = lambda a: torch.tensor(np.asarray(a, np.float32), device="cuda:0")  # noqa: E731
    x = np.linspace(-740.0, 740.0, nlam)
    n = per_sm * (sms or torch.cuda.get_device_properties(0).multi_processor_count) + 3
    p = W.quiet_and_active_params(n, 510 + per_sm)
    tf, tx = t(W.hmi_filters(x)), t(x)
    out = []
    for block in (128, 384):
        h = v.vfisv_create(0)
        if not out:
            syn = v.vfisv_synth(h, t(p), tf, tx, LINE).reshape(n, 24)
            sig = 1e-3 * t(W.continuum(p))[:, None]
            obs = (syn + sig * t(W.noise(n, 24, 510))).contiguous()
            w = (1.0 / (sig * sig)).expand(n, 24).contiguous()
            obs[1, 3] = float("nan")
        v.vfisv_set_launch_shape(h, block, 1)
        v.vfisv_set_sm_limit(h, sms)
        r = v.vfisv_invert(h, obs, w, tf, tx, LINE)
        v.vfisv_check(h)
        out.append((r, v.vfisv_counters(h)))
        h.close()
    (a, ca), (b, cb) = out
    for k in a:
        q, r = (z.view(torch.int32) if z.dtype == torch.float32 else z for z in (a[k], b[k]))
        assert torch.equal(q, r), k
    assert ca == cb and cb["retired"] == n - 1, (ca, cb)
