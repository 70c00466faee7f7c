"""The calls this library is used for, as measurable cases.

A case is one call (or the short chain of calls a program always makes
together) through the public binding, on inputs with the distributions of
the workloads: filtergrams of the HMI-like instrument (six filters on 149
points around Fe I 6173 A) and spectra of the 112-sample spectrograph
(Fe I 6302.5 A).  Inputs are synthesised here in plain torch from the seed
alone, so they do not depend on the code that is measured.

Kinds:
  invert   vfisv_invert of one map
  mixed    vfisv_invert_nn: network guess, confidence routing, re-inversion
  batch    vfisv_invert_batch of many uneven maps (filtergrams start from the
           network's guess, spectra from their weak-field models)
  synth    vfisv_synth
  train    vfisv_nn_train, one epoch from fresh weights
  infer    vfisv_nn_infer
  prep     vfisv_limb_weights and vfisv_init_models of one map
"""
import functools
import math

import numpy as np
import torch

import paper_0901_2702_gb300 as vf

DEV = "cuda:0"
FE6173 = {"lambda0_A": 6173.34, "geff": 2.5, "mu": 1.0}
FE6302 = {"lambda0_A": 6302.4936, "geff": 2.5, "mu": 1.0}
CENTRES = (-172.5, -103.5, -34.5, 34.5, 103.5, 172.5)
DEG = math.pi / 180.0


def listed():
    return [
        # a small patch while looking at a map: the call's latency
        {"name": "invert_patch_300", "kind": "invert", "npix": 300, "sky": "mix", "cov": True},
        # a 64 x 64 cut-out with its error bars
        {"name": "invert_64x64", "kind": "invert", "npix": 4096, "sky": "mix", "cov": True},
        # a 1024 x 1024 map, plain LM from the standard guess, as the library comes
        {"name": "invert_1024x1024", "kind": "invert", "npix": 1048576, "sky": "mix", "cov": True},
        # a disk of 2048 x 2048 (the largest maps served), 90 % quiet Sun, the
        # network-initialised inversion with the launch shape that the
        # autotuner takes on such maps
        {"name": "mixed_disk_2048", "kind": "mixed", "side": 2048, "cov": True, "block": 384},
        # the serving mix: uneven maps in one launch, both instruments
        {"name": "batch_filtergrams", "kind": "batch", "instr": "hmi", "nmaps": 16, "side_min": 32,
         "side_max": 512, "cov": True, "block": 384},
        {"name": "batch_spectra", "kind": "batch", "instr": "spec", "nmaps": 16, "side_min": 32,
         "side_max": 160, "cov": True, "block": 0},
        # one slit-scan patch of spectra, plain LM from the standard guess
        {"name": "invert_spectra_48x48", "kind": "invert", "instr": "spec", "npix": 2304, "sky": "mix",
         "cov": True},
        # training profiles
        {"name": "synth_1m", "kind": "synth", "npix": 1048576, "nf": 6},
        {"name": "synth_spectra_64k", "kind": "synth", "instr": "spec", "npix": 65536},
        # sixteen Adam steps of the workload's batch
        {"name": "train_16_steps", "kind": "train", "npix": 131072, "batch": 8192},
        # initial models of a 1024 x 1024 map
        {"name": "infer_1024x1024", "kind": "infer", "npix": 1048576},
        # weights and weak-field models of a map's filtergrams
        {"name": "prep_1024x1024", "kind": "prep", "npix": 1048576},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more call of the same ranges: sizes over their logarithm, odd ones
    among them, the options that programs set."""
    kind = rng.choice(["invert"] * 4 + ["mixed"] * 2 + ["batch"] * 2 +
                      ["synth", "train", "infer", "prep"])
    instr = "spec" if kind in ("invert", "batch", "synth") and rng.random() < 0.3 else "hmi"
    c = {"kind": kind, "instr": instr}
    if kind == "invert":
        c["npix"] = _log(rng, 1, 60000 if instr == "spec" else 700000)
        c["sky"] = rng.choice(["mix", "quiet"])
        c["cov"] = rng.random() < 0.7
        c["row_weights"] = rng.random() < 0.3  # one weight row for all pixels
        c["weak_field"] = rng.random() < (0.5 if instr == "spec" else 0.2)
        if instr == "hmi":
            c["block"] = rng.choice([0, 0, 384])
            c["nlam"] = rng.choice([75, 149, 149, 297])
            c["free_alpha"] = rng.random() < 0.1
    elif kind == "mixed":
        c.update(side=_log(rng, 32, 1500), cov=rng.random() < 0.7, block=rng.choice([0, 384]))
    elif kind == "batch":
        c.update(nmaps=rng.randint(3, 24), side_min=32, cov=rng.random() < 0.5,
                 side_max=_log(rng, 48, 160 if instr == "spec" else 500),
                 block=0 if instr == "spec" else rng.choice([0, 384]))
    elif kind == "synth":
        c["npix"] = _log(rng, 1, 150000 if instr == "spec" else 4000000)
        if instr == "hmi":
            c["nf"] = rng.choice([1, 4, 6, 6, 8])
            c["nlam"] = rng.choice([75, 149, 149, 297])
            c["mixed_alpha"] = rng.random() < 0.3
    elif kind == "train":
        c["batch"] = 512 * rng.choice([1, 4, 16, 16])
        c["npix"] = c["batch"] * rng.randint(2, 20) + rng.randint(0, 511)
    else:
        c["npix"] = _log(rng, 1, 4000000)
    return c


# ---------------------------------------------------------------------------
# Instruments: filter profiles [nf, nlam] and wavelength offsets [nlam] (mA).


@functools.lru_cache(maxsize=None)
def _instrument(instr, nf=6, nlam=149):
    if instr == "spec":
        n, step = 112, 21.5
        x = (np.arange(4 * n) - (4 * n - 1) / 2.0) * (step / 4)
        d = x[None, :] - ((np.arange(n) - (n - 1) / 2.0) * step)[:, None]
        t = np.exp(-4.0 * math.log(2.0) * d * d / 25.0 ** 2) * (np.abs(d) <= 75.0)
    else:
        x = (np.arange(nlam) - (nlam - 1) / 2.0) * (1480.0 / (nlam - 1))
        c = np.array(CENTRES) if nf == 6 else (np.arange(nf) - (nf - 1) / 2.0) * 69.0
        d = x[None, :] - c[:, None]
        t = np.exp(-4.0 * math.log(2.0) * d * d / 76.0 ** 2) * np.sinc(d / 152.0) ** 2
    t = t / t.sum(1, keepdims=True)
    f32 = lambda a: torch.tensor(a, dtype=torch.float32, device=DEV)  # noqa: E731
    return f32(t), f32(x), FE6302 if instr == "spec" else FE6173


def _case_instrument(case):
    if case.get("instr") == "spec":
        return _instrument("spec")
    return _instrument("hmi", case.get("nf", 6), case.get("nlam", 149))


# ---------------------------------------------------------------------------
# Milne-Eddington synthesis in plain torch, in the precision of `params`.


@functools.lru_cache(maxsize=None)
def _weideman(n):
    """Coefficients of Weideman's (1994) rational series of w(z) with n terms."""
    L = math.sqrt(n / math.sqrt(2.0))
    m = 64 * n
    th = -math.pi + 2.0 * math.pi * np.arange(m) / m
    t = L * np.tan(0.5 * th[1:])
    f = np.concatenate([[0.0], (L * L + t * t) * np.exp(-t * t)])
    return L, [float((f * np.cos(k * th)).mean()) for k in range(1, n + 1)]


def _faddeeva(u, a):
    """w(u + i a): real part H (Voigt), imaginary part F (Faraday-Voigt)."""
    L, coef = _weideman(40 if u.dtype == torch.float64 else 16)
    iz = torch.complex((-a).expand_as(u), u)
    q = 1.0 / (L - iz)
    Z = (L + iz) * q
    p = torch.full_like(Z, coef[-1])
    for c in reversed(coef[:-1]):
        p = p * Z + c
    w = 2.0 * p * q * q + (1.0 / math.sqrt(math.pi)) * q
    return w.real, w.imag


def _unit_stokes(p, x, line):
    """K^-1 e0 [n, 4, nlam] in the frame of psi = 0."""
    cB = 4.66685e-10 * line["geff"] * line["lambda0_A"] ** 2
    cv = line["lambda0_A"] * 1.0e3 / 299792.458
    B, g, eta0, dl, a, v = (p[:, k, None] for k in (0, 1, 3, 4, 5, 6))
    up = (x[None, :] - cv * v) / dl
    ub = cB * B / dl
    (Hp, Fp), (Hb, Fb), (Hr, Fr) = (_faddeeva(u, a) for u in (up, up + ub, up - ub))
    s2, cg = torch.sin(g * DEG) ** 2, torch.cos(g * DEG)
    c2 = 1 + cg * cg
    eI = 1 + 0.5 * eta0 * (Hp * s2 + 0.5 * (Hb + Hr) * c2)
    eQ, rQ = (0.5 * eta0 * s2 * (k - 0.5 * (b + r)) for k, b, r in ((Hp, Hb, Hr), (Fp, Fb, Fr)))
    eV, rV = 0.5 * eta0 * cg * (Hr - Hb), 0.5 * eta0 * cg * (Fr - Fb)
    pi = eQ * rQ + eV * rV
    e2 = eI * eI
    r2 = rQ * rQ + rV * rV
    D = e2 * (e2 - eQ * eQ - eV * eV + r2) - pi * pi
    return torch.stack([eI * (e2 + r2), -(e2 * eQ + rQ * pi), -eI * (eQ * rV - eV * rQ),
                        -(e2 * eV + rV * pi)], 1) / D[:, None, :]


def _synth(params, T, x, line):
    """Filtered Stokes vector [n, 4, nf] of models [n, 10], in params' precision."""
    T, x = T.to(params.dtype), x.to(params.dtype)
    out = torch.empty((params.shape[0], 4, T.shape[0]), dtype=params.dtype, device=params.device)
    step = max(1, 10000000 // x.numel())
    tau = T.sum(1)
    for i in range(0, params.shape[0], step):
        p = params[i:i + step]
        al = p[:, 9, None, None]
        y = al * (_unit_stokes(p, x, line) @ T.T)
        if bool((p[:, 9] != 1).any()):
            q = p.clone()
            q[:, 0] = 0
            n = _unit_stokes(q, x, line) @ T.T
            y[:, 0] += (1 - al[:, :, 0]) * n[:, 0]
        ps = 2 * DEG * p[:, 2, None]
        c, s = torch.cos(ps), torch.sin(ps)
        m = line["mu"] * p[:, 8, None]
        o = out[i:i + step]
        o[:, 0] = p[:, 7, None] * tau + m * y[:, 0]
        o[:, 1] = m * (c * y[:, 1] - s * y[:, 2])
        o[:, 2] = m * (s * y[:, 1] + c * y[:, 2])
        o[:, 3] = m * y[:, 3]
    return out


# ---------------------------------------------------------------------------
# Models and observations.


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _models(n, g, b_max):
    """Model parameters [n, 10] with the workloads' uniform distributions."""
    u = torch.rand((n, 9), generator=g, device=DEV)
    p = torch.empty((n, 10), device=DEV)
    p[:, 0] = b_max * u[:, 0]
    p[:, 1] = torch.acos(2 * u[:, 1] - 1) / DEG
    p[:, 2] = 180 * u[:, 2]
    p[:, 3] = torch.exp(math.log(50.0) * u[:, 3])
    p[:, 4] = 20 + 30 * u[:, 4]
    p[:, 5] = 0.5 * u[:, 5]
    p[:, 6] = (1.5 * torch.randn(n, generator=g, device=DEV)).clamp(-7, 7)
    p[:, 7] = 0.1 + 0.3 * u[:, 7]
    p[:, 8] = 0.6 + 0.3 * u[:, 8]
    p[:, 9] = 1
    return p


def _disk_models(side, g):
    """A disk of quiet Sun with active regions (field up to 3.5 kG, smooth
    inclination and azimuth) over a tenth of it."""
    ax = torch.arange(side, device=DEV, dtype=torch.float32) - (side - 1) / 2.0
    yy, xx = torch.meshgrid(ax, ax, indexing="ij")
    on = (xx * xx + yy * yy <= (0.5 * side - 0.5) ** 2).reshape(-1).nonzero()[:, 0]
    x, y = xx.reshape(-1)[on], yy.reshape(-1)[on]
    p = _models(x.numel(), g, 200.0)
    best = torch.zeros_like(x)
    for _ in range(64):
        r, th, sig, peak, up = torch.rand(5, generator=g, device=DEV).tolist()
        r = 0.5 * side * math.sqrt(0.9 * r)
        dx, dy = x - r * math.cos(2 * math.pi * th), y - r * math.sin(2 * math.pi * th)
        sig = (64 + 192 * sig) * min(1.0, side / 1024.0) / 2.355
        w = torch.exp(-(dx * dx + dy * dy) / (2 * sig * sig))
        k = w > best.clamp(min=1e-3)
        best = torch.where(k, w, best)
        gc = 0.0 if up < 0.5 else 180.0
        p[:, 0] = torch.where(k, torch.maximum(p[:, 0], (1500 + 2000 * peak) * w), p[:, 0])
        p[:, 1] = torch.where(k, 90 - (90 - gc) * w, p[:, 1])
        p[:, 2] = torch.where(k, torch.remainder(torch.atan2(dy, dx) / DEG, 180.0), p[:, 2])
        if float((best > 0.5).float().mean()) >= 0.1:
            break
    return p


def _observe(p, T, x, line, g, sigma=1e-3):
    """Observed samples [n, 4 nf] with noise of sigma * Ic, and that noise [n, 1]."""
    s = _synth(p, T, x, line).reshape(p.shape[0], -1)
    sig = sigma * (p[:, 7] + line["mu"] * p[:, 8])[:, None]
    return (s + sig * torch.randn(s.shape, generator=g, device=DEV)).contiguous(), sig


# ---------------------------------------------------------------------------
# The network that a program keeps: 24-256-256-256-11, flat float32 blob
# W0 b0 W1 b1 W2 b2 W3 b3 in_mean in_std out_mean out_std.

SIZES = (24, 256, 256, 256, 11)


def _targets(p, ic):
    ps = 2 * DEG * p[:, 2]
    return torch.stack([p[:, 0], torch.cos(DEG * p[:, 1]), torch.sin(ps), torch.cos(ps),
                        torch.log(p[:, 3]), p[:, 4], p[:, 5], p[:, 6], p[:, 7] / ic,
                        p[:, 8] / ic], 1)


def _fresh_blob(obs, p, g):
    """Random weights, zero biases, the training set's statistics."""
    parts = []
    for i, o in zip(SIZES[:-1], SIZES[1:]):
        parts += [(2 * torch.rand((i, o), generator=g, device=DEV) - 1) * math.sqrt(6.0 / i),
                  torch.zeros(o, device=DEV)]
    ic = obs[:, :6].amax(1)
    f, t = obs / ic[:, None], _targets(p, ic)
    parts += [f.mean(0), f.std(0, False), t.mean(0), t.std(0, False)]
    return torch.cat([q.reshape(-1) for q in parts])


def _split_blob(blob):
    layers, at = [], 0
    for i, o in zip(SIZES[:-1], SIZES[1:]):
        layers.append((blob[at:at + i * o].view(i, o), blob[at + i * o:at + i * o + o]))
        at += i * o + o
    stats = []
    for n in (24, 24, 10, 10):
        stats.append(blob[at:at + n])
        at += n
    return layers, stats


def _network(layers, h):
    for k, (W, b) in enumerate(layers):
        h = h @ W + b
        if k < 3:
            h = torch.nn.functional.gelu(h)
    return h


def _loss(layers, stats, obs, p):
    ic = obs[:, :6].amax(1).clamp(min=1e-30)
    y = _network(layers, (obs / ic[:, None] - stats[0]) / stats[1])
    e = ((y[:, :10] - (_targets(p, ic) - stats[2]) / stats[3]) ** 2).mean(1)
    c = torch.log(e.detach() + 1e-4)
    return e.mean() + ((y[:, 10] - c) ** 2).mean()


def _adam(blob, batches, steps, lr0):
    """Adam with cosine decay over `batches` of (obs, params); the losses."""
    n = sum(i * o + o for i, o in zip(SIZES[:-1], SIZES[1:]))
    w = blob[:n].clone()
    m, v = torch.zeros_like(w), torch.zeros_like(w)
    losses = []
    for t, (o, p) in enumerate(batches):
        w = w.detach().requires_grad_(True)
        layers, stats = _split_blob(torch.cat([w, blob[n:]]))
        loss = _loss(layers, stats, o, p)
        g, = torch.autograd.grad(loss, w)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        lr = lr0 * 0.5 * (1 + math.cos(math.pi * t / steps))
        w = w.detach() - lr * (m / (1 - 0.9 ** (t + 1))) / (torch.sqrt(v / (1 - 0.999 ** (t + 1))) + 1e-8)
        losses.append(loss.detach())
    return torch.cat([w.detach(), blob[n:]]), torch.stack(losses)


@functools.lru_cache(maxsize=None)
def _trained_blob():
    """The program's trained network: the same for all its maps."""
    g = _gen(3)
    T, x, line = _instrument("hmi")
    n, batch, steps = 1 << 20, 8192, 1500
    p = _models(n, g, 3000.0)
    obs, _ = _observe(p, T, x, line, g)
    blob = _fresh_blob(obs, p, g)
    batches = ((obs[i:i + batch], p[i:i + batch]) for i in
               ((t * batch) % n for t in range(steps)))
    return _adam(blob, batches, steps, 1e-3)[0].contiguous()


# ---------------------------------------------------------------------------


def _sides(case):
    """Sides of a batch's maps, log-uniform, smallest first (the order in
    which the serving queue holds them)."""
    k, lo, hi = case["nmaps"], case["side_min"], case["side_max"]
    return [int(round(lo * (hi / lo) ** (i / max(1, k - 1)))) for i in range(k)]


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    T, x, line = _case_instrument(case)
    s = {"case": case, "T": T, "x": x, "line": line, "h": vf.vfisv_create(0)}
    if case.get("block"):
        vf.vfisv_set_launch_shape(s["h"], case["block"], 1)
    if kind == "batch":
        parts, rows, off = [], [], [0]
        for side in _sides(case):
            p = _disk_models(side, g)
            rel = 3e-4 * 10.0 ** float(torch.rand(1, generator=g, device=DEV))
            o, _ = _observe(p, T, x, line, g, rel)
            parts.append(o)
            rows.append(torch.full((o.shape[1],), 1.0 / rel ** 2, device=DEV))
            off.append(off[-1] + p.shape[0])
        s.update(obs=torch.cat(parts), w=torch.stack(rows), off=np.array(off, dtype=np.int64))
        if case.get("instr") != "spec":
            s["blob"] = _trained_blob()
        return s
    if kind == "mixed":
        p = _disk_models(case["side"], g)
    else:
        p = _models(case["npix"], g, 200.0 if case.get("sky") == "quiet" else 3000.0)
    if case.get("free_alpha") or case.get("mixed_alpha"):
        p[:, 9] = 0.2 + 0.8 * torch.rand(p.shape[0], generator=g, device=DEV)
    if kind == "synth":
        s["params"] = p
        return s
    obs, sig = _observe(p, T, x, line, g)
    s["obs"] = obs
    if kind in ("invert", "mixed"):
        if case.get("row_weights"):
            s["w"] = torch.full((obs.shape[1],), 1e6, device=DEV)
        else:
            s["w"] = (1.0 / (sig * sig)).expand_as(obs).contiguous()
    if kind in ("mixed", "infer"):
        s["blob"] = _trained_blob()
    if kind == "train":
        s["params"] = p
        s["blob"] = _fresh_blob(obs, p, g)
    if kind == "prep":
        s["mu"] = torch.rand(p.shape[0], generator=g, device=DEV).sqrt()
    return s


SIGMA4 = (1e-3, 1e-3, 1e-3, 1e-3)


def run(s):
    case, h, T, x, line = s["case"], s["h"], s["T"], s["x"], s["line"]
    kind = case["kind"]
    if kind == "invert":
        cfg = {}
        if case.get("weak_field"):
            cfg["wfa_pol"] = 1.0
        if case.get("free_alpha"):
            cfg["free_mask"] = 0x3FF
        return vf.vfisv_invert(h, s["obs"], s["w"], T, x, line, config=cfg, want_cov=case["cov"])
    if kind == "mixed":
        return vf.vfisv_invert_nn(h, s["blob"], s["obs"], s["w"], T, x, line,
                                  config_nn={"max_iter": 50}, chi2_flag=2.5, conf_route=-1.5,
                                  want_cov=case["cov"])
    if kind == "batch":
        if "blob" in s:
            init = vf.vfisv_nn_infer(h, s["blob"], s["obs"], line, want_conf=False)["init"]
            r = vf.vfisv_invert_batch(h, s["obs"], s["w"], s["off"], T, x, line, init=init,
                                      want_cov=case["cov"])
        else:
            r = vf.vfisv_invert_batch(h, s["obs"], s["w"], s["off"], T, x, line,
                                      config={"wfa_pol": 1.0}, want_cov=case["cov"])
        r.pop("latency_ms")  # a measured time, not a result
        return r
    if kind == "synth":
        return vf.vfisv_synth(h, s["params"], T, x, line)
    if kind == "train":
        blob = s["blob"].clone()
        loss = vf.vfisv_nn_train(h, blob, s["obs"], s["params"], batch=case["batch"], epochs=1, seed=3)
        return {"blob": blob, "loss": loss}
    if kind == "infer":
        return vf.vfisv_nn_infer(h, s["blob"], s["obs"], line, want_conf=True, want_raw=True)
    w = vf.vfisv_limb_weights(h, s["obs"], s["mu"], 1.0, SIGMA4)
    m = vf.vfisv_init_models(h, s["obs"], T, x, line)
    return {"w": w, "init": m["init"], "pol": m["pol"]}


# Work per wavelength point of one trial model (an FMA counts twice): 505 for
# the synthesis, 643 for the derivatives, of which only accepted trials (about
# half) need the latter; 63 of 149 points carry the filters' weight.  LM takes
# about 34 trials a pixel on the mixed sky, 37 on the disk, 16 for spectra that
# start from their weak-field models and 27 for those that do not.
def work(case):
    kind = case["kind"]
    spec = case.get("instr") == "spec"
    nf = 112 if spec else case.get("nf", 6)
    pts = 448 if spec else 63 * case.get("nlam", 149) / 149.0
    if kind == "batch":
        n = sum(math.pi * (0.5 * k) ** 2 for k in _sides(case))
    elif kind == "mixed":
        n = math.pi * (0.5 * case["side"]) ** 2
    else:
        n = case["npix"]
    row = 16.0 * nf
    if kind in ("invert", "mixed", "batch"):
        trials = (16 if kind == "batch" or case.get("weak_field") else 27) if spec else \
            34 if kind == "invert" else 37
        b = n * (row + 52 + (400 if case["cov"] else 0))
        if kind != "batch" and not case.get("row_weights"):
            b += n * row
        per = pts * (505 + 0.5 * 643) + 0.5 * 4 * nf * 147
        return {"bytes": b, "flops": n * trials * per}
    if kind == "synth":
        return {"bytes": n * (40 + row), "flops": n * pts * 505}
    if kind == "train":
        steps = n // case["batch"]
        return {"bytes": steps * case["batch"] * 136.0 + 2 * 563516.0,
                "flops": steps * case["batch"] * 827904.0}
    if kind == "infer":
        return {"bytes": n * (96.0 + 40 + 4 + 44), "flops": n * 280064.0}
    return {"bytes": n * (96.0 + 4 + 96 + 40 + 4), "flops": n * 300.0}


# ---------------------------------------------------------------------------
# The same results in 64 bits.


def _decode(y, ic, mu, stats):
    t = y[:, :10] * stats[3] + stats[2]
    ps = torch.remainder(torch.atan2(t[:, 2], t[:, 3]) / (2 * DEG), 180.0)
    return torch.stack([t[:, 0].clamp(min=0), torch.acos(t[:, 1].clamp(-1, 1)) / DEG, ps,
                        torch.exp(t[:, 4]), t[:, 5], t[:, 6], t[:, 7], t[:, 8] * ic,
                        t[:, 9] * ic / mu, torch.ones_like(ic)], 1)


def _weak_field(obs, T, x, line):
    """Weak-field B and gamma, wing azimuth, centre-of-gravity velocity, the
    standard guess for the rest; and the polarisation level."""
    T, x = T.double(), x.double()
    c = (T @ x) / T.sum(1)
    I, Q, U, V = obs.view(-1, 4, T.shape[0]).unbind(1)  # the centres increase
    d1 = torch.empty_like(I)
    d1[:, 0] = (I[:, 1] - I[:, 0]) / (c[1] - c[0])
    d1[:, -1] = (I[:, -1] - I[:, -2]) / (c[-1] - c[-2])
    d1[:, 1:-1] = (I[:, 2:] - I[:, :-2]) / (c[2:] - c[:-2])
    sl = (I[:, 1:] - I[:, :-1]) / (c[1:] - c[:-1])
    d2 = 2 * (sl[:, 1:] - sl[:, :-1]) / (c[2:] - c[:-2])
    C = 4.66685e-10 * line["geff"] * line["lambda0_A"] ** 2
    bpar = -(V * d1).sum(1) / ((d1 * d1).sum(1) * C)
    s22 = (d2 * d2).sum(1)
    qa, ub = (Q[:, 1:-1] * d2).sum(1) / s22, (U[:, 1:-1] * d2).sum(1) / s22
    bperp = 2 * (qa * qa + ub * ub) ** 0.25 / C
    wing = (c - c.mean()) ** 4
    psi = torch.remainder(0.5 * torch.atan2((U * wing).sum(1), (Q * wing).sum(1)) / DEG, 180.0)
    ic = I.amax(1)
    pol = (Q * Q + U * U + V * V).sqrt().amax(1) / ic
    dep = ic[:, None] - I
    v = (dep * c).sum(1) / dep.sum(1) / (line["lambda0_A"] * 1.0e3 / 299792.458)
    one = torch.ones_like(ic)
    m = torch.stack([torch.hypot(bpar, bperp).clamp(max=6000.0), torch.atan2(bperp, bpar) / DEG, psi,
                     10 * one, 35 * one, 0.25 * one, v.clamp(-20, 20), (0.25 * ic).clamp(0, 2),
                     (0.75 * ic / line["mu"]).clamp(0, 2), one], 1)
    return m, pol


def _epoch_order(n, seed):
    """The sample order of the first epoch: k -> (mult k + add) mod n, keyed by the seed."""
    mask = (1 << 64) - 1
    h = (seed * 0x9E3779B97F4A7C15 + 1) & mask
    h ^= h >> 31
    h = (h * 0xBF58476D1CE4E5B9) & mask
    h ^= h >> 29
    mult = 1 + h % (n - 1)
    while math.gcd(mult, n) != 1:
        mult = mult % (n - 1) + 1
    add = (h >> 17) % n
    return torch.tensor([(mult * k + add) % n for k in range(n)], device=DEV)


def exact(case, seed):
    """The results in 64 bits.  The inversions have none: an LM trajectory
    branches at every acceptance test, so on ill-determined pixels one in 64
    bits ends at another point of a flat valley."""
    kind = case["kind"]
    if kind in ("invert", "mixed", "batch"):
        return None
    s = prepare(case, seed)
    T, x, line = s["T"], s["x"], s["line"]
    if kind == "synth":
        return _synth(s["params"].double(), T, x, line)
    obs = s["obs"].double()
    if kind == "train":
        n, b = case["npix"], case["batch"]
        o = _epoch_order(n, 3)
        steps = n // b
        p = s["params"].double()
        batches = ((obs[o[t * b:(t + 1) * b]], p[o[t * b:(t + 1) * b]]) for t in range(steps))
        blob, loss = _adam(s["blob"].double(), batches, steps, 1e-3)
        return {"blob": blob, "loss": loss}
    if kind == "infer":
        layers, stats = _split_blob(s["blob"].double())
        ic = obs[:, :6].amax(1)
        y = torch.cat([_network(layers, (o / o[:, :6].amax(1, keepdim=True) - stats[0]) / stats[1])
                       for o in obs.split(1 << 17)])
        return {"init": _decode(y, ic, line["mu"], stats), "conf": y[:, 10].contiguous(), "raw": y}
    ic = obs[:, :6].amax(1)
    mu = s["mu"].double()
    limb = 0.33644 + mu * (1.30590 + mu * (-1.79238 + mu * (2.45050 + mu * (-1.89979 + mu * 0.59943))))
    w = torch.full_like(obs, 1e6)
    w[:, :6] *= ((0.7778 * (limb - ic).abs() + 0.3) ** 2)[:, None]
    m, pol = _weak_field(obs, T, x, line)
    return {"w": w, "init": m, "pol": pol}
