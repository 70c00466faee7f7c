"""The LM kernel with eight lanes per pixel, which a handle without a launch
shape runs on small maps, against the one-warpgroup kernel (128 x 1): the same
operations and sums in the same order, so every output and the work counters
agree bit for bit.  Sizes around its warps of four pixels and its queue
(more pixels than are resident), bad input pixels, initial models, caps 0 and
1, Hessian reuse, held parameters (the solve's held rows), nearly singular
pixels (the solve's one-lane fallback), grids whose kept points fill the last
step of eight or leave one over, shared weights, batched maps, the mixed
inversion's pixel list, an SM limit, and a replayed graph."""
import numpy as np
import pytest

import workloads as W
from gpu_common import LINE, T, X, vf  # noqa: F401

pytestmark = pytest.mark.gpu


def _map(v, h, torch, n, seed, T_=T, X_=X, b_max=3000.0):
    t = lambda a: torch.tensor(np.asarray(a, np.float32), device="cuda:0")  # noqa: E731
    p = W.quiet_and_active_params(n, seed, b_max=b_max)
    tf, tx = t(T_), t(X_)
    syn = v.vfisv_synth(h, t(p), tf, tx, LINE).reshape(n, 24)
    sig = 1e-3 * t(W.continuum(p))[:, None]
    obs = (syn + sig * t(W.noise(n, 24, seed))).contiguous()
    return p, obs, (1.0 / (sig * sig)).expand(n, 24).contiguous(), tf, tx


@pytest.fixture()
def pair(vf):
    """(library, torch, handle without a shape, handle set to 128 x 1)."""
    v, _, torch = vf
    a, b = v.vfisv_create(0), v.vfisv_create(0)
    v.vfisv_set_launch_shape(b, 128, 1)
    yield v, torch, a, b
    a.close()
    b.close()


def _equal(v, torch, a, b, call):
    out = []
    for h in (a, b):
        v.vfisv_counters(h, reset=True)
        r = call(h)
        v.vfisv_check(h)
        out.append((r, v.vfisv_counters(h, reset=True)))
    (ra, ca), (rb, cb) = out
    for k in ra:
        if ra[k] is None or k == "latency_ms":
            continue
        x, y = (z.view(torch.int32) if z.dtype == torch.float32 else z for z in (ra[k], rb[k]))
        assert torch.equal(x, y), k
    assert ca == cb, (ca, cb)
    return ra


@pytest.mark.parametrize("n", [1, 3, 5, 300, 2433, 12001])
def test_same_bits(pair, n):
    v, torch, a, b = pair
    p, obs, w, tf, tx = _map(v, a, torch, n, 40 + n)
    if n > 3:
        obs[1, 3] = float("nan")
        w[2] = 0.0
    r = _equal(v, torch, a, b, lambda h: v.vfisv_invert(h, obs, w, tf, tx, LINE))
    if n > 3:
        assert r["status"][1:3].tolist() == [3, 3]


@pytest.mark.parametrize("cfg", [{"max_iter": 0}, {"max_iter": 1}, {"hess_reuse": 1e-2},
                                 {"free_mask": 0x0F7}, {"free_mask": 0x1F8}, {"wfa_pol": 1.0},
                                 {"eps0": 1e-9, "conv_eps": 10.0}])
def test_same_bits_with_options(pair, cfg):
    v, torch, a, b = pair
    n = 1500
    p, obs, w, tf, tx = _map(v, a, torch, n, 78, b_max=1e-2 if "eps0" in cfg else 3000.0)
    init = None
    if "wfa_pol" not in cfg:
        init = torch.tensor(np.asarray(p, np.float32), device="cuda:0")
        init[:, 3] *= 0.8
    _equal(v, torch, a, b, lambda h: v.vfisv_invert(h, obs, w[0].contiguous(), tf, tx, LINE,
                                                    init=init, config=cfg))


@pytest.mark.parametrize("nlam", [1, 8, 9, 37, 600])
def test_same_bits_on_other_grids(pair, nlam):
    v, torch, a, b = pair
    x = np.linspace(-600.0, 650.0, nlam) if nlam > 1 else np.zeros(1)
    p, obs, w, tf, tx = _map(v, a, torch, 700, nlam, T_=W.hmi_filters(x), X_=x)
    _equal(v, torch, a, b, lambda h: v.vfisv_invert(h, obs, w, tf, tx, LINE))


def test_same_bits_batched_mixed_and_limited(pair):
    v, torch, a, b = pair
    sizes = [1, 700, 33, 2000, 129]
    parts = [_map(v, a, torch, n, 900 + i) for i, n in enumerate(sizes)]
    obs = torch.cat([q[1] for q in parts]).contiguous()
    wm = torch.stack([q[2][0] * (1.0 + 0.1 * i) for i, q in enumerate(parts)]).contiguous()
    tf, tx = parts[0][3], parts[0][4]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    r = _equal(v, torch, a, b, lambda h: v.vfisv_invert_batch(h, obs, wm, off, tf, tx, LINE))
    assert bool((r["latency_ms"] > 0).all())
    p = torch.tensor(np.concatenate([q[0] for q in parts]).astype(np.float32), device="cuda:0")
    w = torch.cat([q[2] for q in parts]).contiguous()
    blob = v.vfisv_nn_init(a, obs, p, seed=5)
    k = float(v.vfisv_nn_infer(a, blob, obs, LINE)["conf"].median().item())
    _equal(v, torch, a, b, lambda h: v.vfisv_invert_nn(h, blob, obs, w, tf, tx, LINE,
                                                       conf_route=k))
    v.vfisv_set_sm_limit(a, 19)
    _equal(v, torch, a, b, lambda h: v.vfisv_invert(h, obs[:1000], w[:1000], tf, tx, LINE))
    v.vfisv_set_sm_limit(a, 0)


def test_same_bits_in_a_replayed_graph(pair):
    v, torch, a, b = pair
    n = 900
    _, obs, w, tf, tx = _map(v, a, torch, n, 71)
    _, obs2, _, _, _ = _map(v, a, torch, n, 72)
    s = torch.cuda.Stream(torch.device("cuda:0"))
    src = obs.clone()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        out = v.vfisv_invert(a, src, w, tf, tx, LINE, stream=s)  # sizes the workspaces
        s.synchronize()
        v.vfisv_graph_begin(a, s)
        v.vfisv_invert(a, src, w, tf, tx, LINE, out=out, stream=s)
        g = v.vfisv_graph_end(a, s)
        for data in (obs, obs2):
            src.copy_(data)
            g.launch(s)
            s.synchronize()
            ref = v.vfisv_invert(b, data, w, tf, tx, LINE, stream=s)
            s.synchronize()
            for k in out:
                assert torch.equal(out[k], ref[k]), k
    g.close()


@pytest.mark.parametrize("nlam,per_sm", [(160, 85), (160, 128), (161, 128), (230, 256),
                                         (231, 256), (320, 300), (321, 300), (400, 640),
                                         (401, 640)])
@pytest.mark.parametrize("extra", [0, 1])
def test_same_bits_at_the_lines_of_the_rule(pair, nlam, per_sm, extra):
    # pixels an SM and wavelength points where the kernel chosen changes
    v, torch, a, b = pair
    n = 8 * per_sm + extra
    x = np.linspace(-740.0, 740.0, nlam)
    p, obs, w, tf, tx = _map(v, a, torch, n, nlam + n, T_=W.hmi_filters(x), X_=x)
    v.vfisv_set_sm_limit(a, 8)
    _equal(v, torch, a, b, lambda h: v.vfisv_invert(h, obs, w, tf, tx, LINE))
