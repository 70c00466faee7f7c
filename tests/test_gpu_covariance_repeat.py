"""Singular pixels' covariance over repeated calls: which of the eigen
fallback's two paths (one pixel a lane, or a group of lanes) a pixel takes goes
by its place in a queue that atomics fill, so a row's bits may not depend on
the path, on the same map and among other pixels alike."""
import numpy as np
import pytest

import workloads as W
from gpu_common import LINE, T, X, vf  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [12, 700, 12000])
@pytest.mark.parametrize("mask,fast", [(0x1FF, 0), (0x1FF, 1), (0x1F7, 0), (0x3FF, 0)])
def test_repeated_calls_give_the_same_bits(vf, n, mask, fast):  # noqa: F811
    v, h, torch = vf
    t = lambda a: torch.tensor(np.asarray(a, np.float32), device="cuda:0")  # noqa: E731
    p = W.quiet_and_active_params(n, 83, b_max=1e-3)
    p[::3, 0] *= 1e5
    tf, tx = t(T), t(X)
    obs = v.vfisv_synth(h, t(p), tf, tx, LINE).reshape(n, 24) + 1e-3 * t(W.noise(n, 24, 83))
    w = torch.full((24,), 1e6, device="cuda:0")
    init = t(p)
    cfg = {"max_iter": 0, "free_mask": mask, "fast_solve": fast}

    def cov(q):
        r = v.vfisv_invert(h, obs[q].contiguous(), w, tf, tx, LINE, init=init[q].contiguous(),
                           config=cfg)
        return r["cov"].view(torch.int32)  # bits: some variances leave FP32's range

    rows = torch.arange(n, device="cuda:0")
    first = cov(rows)
    for _ in range(4):
        assert torch.equal(cov(rows), first)
    # other neighbours: the rows in reverse, and every second one of them
    assert torch.equal(cov(rows.flip(0)), first.flip(0))
    assert torch.equal(cov(rows[::2]), first[::2])
    v.vfisv_check(h)
