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


def _ms(torch, call, reps=6):
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = float("inf")
    for i in range(reps):
        a.record()
        call()
        b.record()
        b.synchronize()
        if i:
            best = min(best, a.elapsed_time(b))
    return best


# points of the grid, half its span (mA; the filters end at 310: nothing beyond
# is kept), pixels an SM, most that the call may take of 128 x 1's time
@pytest.mark.parametrize("nlam,half,per_sm,most", [
    (80, 310.0, 110, 1.1), (149, 310.0, 257, 1.1), (230, 310.0, 258, 1.1), (190, 310.0, 640, 1.1),
    (600, 310.0, 256, 1.1), (2500, 310.0, 150, 1.1), (3000, 14500.0, 129, 1.1),
    # few points kept: the warp-specialised kernel's gain has to stay
    (149, 740.0, 200, 0.9), (600, 2900.0, 257, 0.95), (1700, 8300.0, 256, 0.85)])
def test_the_choice_goes_by_the_points_kept(vf, nlam, half, per_sm, most):  # noqa: F811
    """A pass costs the grid points that the filter table keeps, not those of
    the grid: on grids cut to the filters' support as on wide ones, a call
    without a set shape is no slower than 128 x 1, and the same bits (margin:
    10 %; choosing by the grid's points lost up to 57 % here)."""
    v, _, torch = vf
    a, b = v.vfisv_create(0), v.vfisv_create(0)
    v.vfisv_set_launch_shape(b, 128, 1)
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    obs, w, tf, tx = _map(v, a, torch, n, np.linspace(-half, half, nlam))
    out = [v.vfisv_invert(h, obs, w, tf, tx, LINE, want_cov=False) for h in (a, b)]
    for k in out[0]:
        assert out[0][k] is None or torch.equal(out[0][k], out[1][k]), k
    ms = [_ms(torch, lambda: v.vfisv_invert(h, obs, w, tf, tx, LINE, want_cov=False, out=o))
          for h, o in zip((a, b), out)]
    print(f"{nlam} points to {half} mA, {per_sm} pixels an SM: {ms[0]:.2f} / {ms[1]:.2f} ms")
    assert ms[0] <= most * ms[1], ms
    for h in (a, b):
        v.vfisv_check(h)
        h.close()


X149 = np.linspace(-740.0, 740.0, 149)


@pytest.mark.parametrize("n", [1, 300, 4096])
def test_autotune_of_a_small_map_is_no_loss(vf, n):  # noqa: F811
    """The kernel that small maps take without a set shape is a candidate of the
    autotuner, so a tuned handle is no slower on its sample than an untouched
    one (1.2 ms against 3.7 on 300 pixels when it was not)."""
    v, _, torch = vf
    a, b = v.vfisv_create(0), v.vfisv_create(0)
    obs, w, tf, tx = _map(v, a, torch, n, X149)
    shape = v.vfisv_autotune(b, obs, w, tf, tx, LINE)
    assert shape[:2] == (0, 1) and len(shape[2]) == 10 and all(m > 0 for m in shape[2])
    out = [v.vfisv_invert(h, obs, w, tf, tx, LINE, want_cov=False) for h in (a, b)]
    for k in out[0]:
        assert out[0][k] is None or torch.equal(out[0][k], out[1][k]), k
    ms = [_ms(torch, lambda: v.vfisv_invert(h, obs, w, tf, tx, LINE, want_cov=False, out=o))
          for h, o in zip((a, b), out)]
    assert ms[1] <= 1.1 * ms[0], ms
    for h in (a, b):
        v.vfisv_check(h)
        h.close()


def test_shapes_are_given_back(vf):  # noqa: F811
    """A failed autotuning run leaves the handle's shape alone, and 0 x 1 takes a
    set one off.  Four threads a pixel sum in another order, so their results
    tell whether the shape is still set."""
    v, _, torch = vf
    a, b = v.vfisv_create(0), v.vfisv_create(0)
    obs, w, tf, tx = _map(v, a, torch, 2000, X149)
    call = lambda h: v.vfisv_invert(h, obs, w, tf, tx, LINE, want_cov=False)  # noqa: E731
    plain = call(a)
    v.vfisv_set_launch_shape(b, 128, 4)
    four = call(b)
    same = lambda p, q: all(torch.equal(p[k], q[k]) for k in p if p[k] is not None)  # noqa: E731
    assert not same(plain, four)
    with pytest.raises(v.VfisvError):
        v.vfisv_autotune(b, obs, w, tf, tx, LINE, config={"max_iter": -1})
    assert same(call(b), four)
    v.vfisv_set_launch_shape(b, 0, 1)
    assert same(call(b), plain)
    ms = [_ms(torch, lambda: call(h)) for h in (a, b)]
    v.vfisv_set_launch_shape(b, 128, 1)
    assert max(ms) < 0.7 * _ms(torch, lambda: call(b)), ms  # the eight-lane kernel again
    for tpp in (0, 2, 4):
        with pytest.raises(v.VfisvError):
            v.vfisv_set_launch_shape(b, 0, tpp)
    for h in (a, b):
        v.vfisv_check(h)
        h.close()
