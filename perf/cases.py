"""Performance cases of the finite-difference sweep: what users of the library have it do.

Every case is a whole call (or a short sequence of calls) through the package's public
entry points on synthetic models of the sizes that the workloads, tests and benchmark of
this repository use: single shots on small and large grids, odd-sized grids with several
shots and a 3-D absorbing mask, binary16 storage, TTI at the paper's space orders, the
adjoint, the FWI gradient through autograd and the serving engine.  ``exact`` restates
each of them in 64 bits with plain torch tensor arithmetic.

Conventions: arrays are [z][y][x]; coordinates (x, y, z) in m; time in ms; km/s.
"""
from __future__ import annotations

import math

import torch

import paper_1807_03032_gb300 as fd
from paper_1807_03032_gb300.autograd import acoustic_modeling
from paper_1807_03032_gb300.serving import Engine

H = 20.0          # grid spacing [m]
V_MIN, V_MAX = 1.5, 4.5
EPS_MAX = 0.3     # largest Thomsen epsilon of the TTI models
F0 = 0.010        # Ricker peak frequency [kHz]


# ---------------------------------------------------------------- the cases

def _forward(name, so, shape, nt, shots=1, nsrc=1, rec=64, border=10, mask=False, storage="f32",
             final=True):
    return {"name": name, "kind": "forward", "so": so, "nz": shape[0], "ny": shape[1],
            "nx": shape[2], "nt": nt, "shots": shots, "nsrc": nsrc, "rec": rec, "border": border,
            "mask": mask, "storage": storage, "final": final}


def _tti(name, so, shape, nt, shots=1, nsrc=1, rec=64, border=10, deriv="centred", receiver="p",
         final=True):
    return {"name": name, "kind": "tti", "so": so, "nz": shape[0], "ny": shape[1],
            "nx": shape[2], "nt": nt, "shots": shots, "nsrc": nsrc, "rec": rec, "border": border,
            "deriv": deriv, "receiver": receiver, "final": final}


def _inverse(name, kind, so, shape, nt, shots, rec, border=10):
    return {"name": name, "kind": kind, "so": so, "nz": shape[0], "ny": shape[1],
            "nx": shape[2], "nt": nt, "shots": shots, "nsrc": 1, "rec": rec, "border": border}


def listed():
    return [
        # the smallest acoustic workload (a quick look at one shot): launches and latency count
        _forward("acoustic_64_so4", 4, (64, 64, 64), 100),
        # an odd-sized grid with two shots of several simultaneous sources and a 3-D absorbing mask
        _forward("acoustic_ragged_so12_mask", 12, (127, 181, 203), 160, shots=2, nsrc=4, rec=700,
                 border=16, mask=True),
        # one shot of a survey on an ordinary model, receivers at every surface node, wavefield kept
        _forward("acoustic_256_so8", 8, (256, 256, 256), 238, rec=256 * 256, border=40),
        # the benchmark's grid at the widest stencil, traces only (400 ms of propagation)
        _forward("acoustic_512_so16", 16, (512, 512, 512), 238, rec=512 * 512, border=40,
                 final=False),
        # binary16 storage where it is the faster storage (twice the model in the same memory)
        _forward("acoustic_384_so4_f16", 4, (384, 384, 384), 200, rec=384 * 384, border=40,
                 storage="f16"),
        # the smallest TTI workload
        _tti("tti_48_so4", 4, (48, 48, 48), 80, rec=32, border=8),
        # the paper's TTI test at its lowest order
        _tti("tti_384_so4", 4, (384, 384, 384), 60, rec=384 * 384, border=40),
        # the paper's TTI grid at a middle order, traces only
        _tti("tti_512_so8", 8, (512, 512, 512), 60, rec=512 * 512, border=40, final=False),
        # TTI on an odd-sized grid at the widest stencil
        _tti("tti_ragged_so16", 16, (215, 260, 333), 60, nsrc=2, rec=1500, border=20),
        # adjoint of two shots: residual traces back to the sources
        _inverse("adjoint_160_so8", "adjoint", 8, (160, 160, 160), 200, 2, 96 * 96, border=16),
        # one FWI evaluation through autograd: traces, gradients of the model and the wavelets
        _inverse("fwi_128_so8", "gradient", 8, (128, 128, 128), 240, 4, 64 * 64, border=16),
        # a served model: eight shots of different lengths stepped together by the batch engine
        _inverse("serve_128_so8", "serve", 8, (128, 128, 128), 240, 8, 128 * 128, border=16),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["forward"] * 5 + ["tti"] * 4 + ["adjoint", "gradient", "serve"])
    so = rng.choice([4, 8, 12, 16])
    top = {"forward": 480, "tti": 400, "adjoint": 240, "gradient": 140, "serve": 140}[kind]
    n = _log_uniform(rng, 44, top)
    if rng.random() < 0.3:  # an even cube, as many models are
        side = max(48, int(n) // 16 * 16)
        shape = (side, side, side)
    else:
        shape = tuple(max(36, int(n * rng.uniform(0.75, 1.25))) for _ in range(3))
    points = shape[0] * shape[1] * shape[2]
    shots = 1 if points > 100 ** 3 and kind in ("forward", "tti") else rng.randint(1, 4)
    if kind == "serve":
        shots = rng.randint(2, 8)
    # points x steps x shots of a drawn case stay below the largest listed ones
    most = {"forward": 2.4e10, "tti": 5.0e9, "adjoint": 1.2e10, "gradient": 3.0e9,
            "serve": 6.0e9}[kind]
    nt = int(_log_uniform(rng, 50, 400 if kind != "tti" else 100))
    nt = max(6, min(nt, int(most / (points * shots))))
    border = rng.choice([8, 10, 16])
    rec = int(_log_uniform(rng, 16, min(60000, shape[1] * shape[2])))
    nsrc = rng.choice([1, 1, 1, 2, 5, 20])
    if kind == "forward":
        option = rng.choice(["f32", "f32", "f32", "mask", "f16", "auto"])
        return _without_name(_forward(
            "", so, shape, nt, shots, nsrc, rec, border, mask=option == "mask",
            storage="f32" if option == "mask" else option, final=rng.random() < 0.6))
    if kind == "tti":
        return _without_name(_tti(
            "", so, shape, nt, shots, nsrc, rec, border,
            deriv=rng.choice(["centred", "centred", "centred", "staggered"]),
            receiver=rng.choice(["p", "p", "mean"]), final=rng.random() < 0.6))
    return _without_name(_inverse("", kind, so, shape, nt, shots, min(rec, 20000), border))


def _without_name(case):
    return {k: v for k, v in case.items() if k != "name"}


# ---------------------------------------------------------------- inputs

def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _smooth(shape, gen, lo, hi, sigma=6.0):
    """Gaussian-filtered white noise (periodic, by FFT), rescaled to [lo, hi]."""
    dev = gen.device
    f = torch.fft.rfftn(torch.randn(shape, generator=gen, device=dev, dtype=torch.float32))
    for ax, n in enumerate(shape):
        k = torch.fft.rfftfreq(n, device=dev) if ax == 2 else torch.fft.fftfreq(n, device=dev)
        g = torch.exp(-2.0 * (math.pi * sigma * k) ** 2)
        f *= g.reshape([-1 if a == ax else 1 for a in range(3)])
    f = torch.fft.irfftn(f, s=shape)
    mn, mx = f.aminmax()
    return (lo + (f - mn) * ((hi - lo) / (mx - mn))).clamp_(lo, hi).contiguous()


def _sponge(n, border, vmax, dev):
    """Quadratic absorbing profile of one axis (1/ms)."""
    d0 = 3.0 * vmax * math.log(1e3) / (2.0 * border * H)
    i = torch.arange(n, device=dev, dtype=torch.float64)
    dist = torch.maximum(border - i, i - (n - 1 - border)).clamp_(min=0.0)
    return d0 * (dist / border) ** 2


def _ricker(t):
    a = (math.pi * F0 * (t - 1.0 / F0)) ** 2
    return (1.0 - 2.0 * a) * torch.exp(-a)


def _inputs(case, seed):
    """All arrays of a case (float32, on the device), from the seed alone."""
    dev = _device()
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) * 7919 + 17)
    shape = (case["nz"], case["ny"], case["nx"])
    shots, nsrc, nt, border = case["shots"], case["nsrc"], case["nt"], case["border"]
    tti = case["kind"] == "tti"
    x = {"m": _smooth(shape, gen, V_MIN, V_MAX).pow_(-2)}
    dt = 0.38 * H / (V_MAX * math.sqrt(1.0 + 2.0 * EPS_MAX) if tti else V_MAX)
    prof = [_sponge(n, border, V_MAX, dev) for n in (case["nx"], case["ny"], case["nz"])]
    if case.get("mask"):  # not separable: the ramps' maximum, modulated by smooth noise
        edge = torch.maximum(torch.maximum(prof[2][:, None, None], prof[1][None, :, None]),
                             prof[0][None, None, :])
        x["damp"] = (edge * _smooth(shape, gen, 0.7, 1.3)).float().contiguous()
    else:
        x["damp"] = torch.cat(prof).float()
    if tti:
        x["eps"] = _smooth(shape, gen, 0.06, EPS_MAX)
        x["delta"] = x["eps"] * _smooth(shape, gen, 0.1, 0.8)
        x["theta"] = _smooth(shape, gen, 0.0, math.pi / 4)
        x["phi"] = _smooth(shape, gen, 0.0, math.pi / 4)
    uniform = lambda *s: torch.rand(s, generator=gen, device=dev, dtype=torch.float64)  # noqa: E731
    size = torch.tensor([case["nx"] - 1, case["ny"] - 1, case["nz"] - 1], device=dev,
                        dtype=torch.float64)
    # sources in the middle half below the top border, receivers half a cell below it
    src = (0.25 + 0.5 * uniform(shots, nsrc, 3)) * size
    src[..., 2] = border + 1.0 + 4.0 * uniform(shots, nsrc)
    x["src_xyz"] = (src * H).float()
    rec = uniform(shots, case["rec"], 3) * size
    side = int(round(math.sqrt(case["rec"])))
    if side * side == case["rec"]:  # a regular surface grid
        gx = torch.linspace(0.0, case["nx"] - 1.0, side, device=dev, dtype=torch.float64)
        gy = torch.linspace(0.0, case["ny"] - 1.0, side, device=dev, dtype=torch.float64)
        rec[..., 0] = gx.repeat(side)
        rec[..., 1] = gy.repeat_interleave(side)
    rec[..., 2] = border + 0.5
    x["rec_xyz"] = (rec * H).float()
    t = torch.arange(nt, device=dev, dtype=torch.float64) * dt
    amp = 0.5 + uniform(shots, nsrc)
    x["src_wav"] = (_ricker(t)[None, :, None] * amp[:, None, :]).float().contiguous()
    if case["kind"] in ("adjoint", "gradient"):
        # observed traces: the direct wave of a 2.5 km/s medium
        obs = torch.empty((shots, nt, case["rec"]), device=dev, dtype=torch.float32)
        for s in range(shots):
            r = (x["rec_xyz"][s].double() - x["src_xyz"][s, 0].double()).norm(dim=-1).clamp_(H)
            obs[s] = (amp[s, 0] * H ** 3 / (4.0 * math.pi * r)
                      * _ricker(t[:, None] - r / 2.5)).float()
        x["obs"] = obs
    if case["kind"] == "serve":  # shots of one model stop at different times
        x["nts"] = [max(2, int(nt * (0.6 + 0.4 * (s + 1) / shots))) for s in range(shots)]
    return x, dt


class _State(dict):
    """A case's arrays and, for a served model, its engine (closed with the state)."""

    def __del__(self):
        if "engine" in self:
            self["engine"].close()


def prepare(case, seed):
    x, dt = _inputs(case, seed)
    shape = (case["nz"], case["ny"], case["nx"])
    st = _State(case=case, x=x, dt=dt, grid=fd.Grid(shape, (H, H, H)))
    if case["kind"] == "gradient":
        x["m"].requires_grad_(True)
        x["src_wav"].requires_grad_(True)
    if case["kind"] == "serve":
        st["engine"] = Engine(st["grid"], case["so"], dt, x["m"], x["damp"], case["shots"],
                              case["nsrc"], case["rec"])
        st["wavs"] = [x["src_wav"][s, :n].contiguous() for s, n in enumerate(x["nts"])]
    return st


def run(st):
    case, x, g, dt = st["case"], st["x"], st["grid"], st["dt"]
    kind, so, nt = case["kind"], case["so"], case["nt"]
    if kind == "forward":
        return fd.acoustic_forward(g, so, dt, nt, x["m"], x["src_xyz"], x["src_wav"],
                                   x["rec_xyz"], damp=x["damp"], return_final=case["final"],
                                   storage=case["storage"],
                                   damp_layout="field" if case["mask"] else "axes")
    if kind == "tti":
        return fd.tti_forward(g, so, dt, nt, x["m"], x["eps"], x["delta"], x["theta"], x["phi"],
                              x["src_xyz"], x["src_wav"], x["rec_xyz"], damp=x["damp"],
                              return_final=case["final"], deriv=case["deriv"],
                              receiver=case["receiver"])
    if kind == "adjoint":
        return fd.acoustic_adjoint(g, so, dt, nt, x["m"], x["src_xyz"], x["rec_xyz"], x["obs"],
                                   damp=x["damp"])
    if kind == "gradient":
        rec = acoustic_modeling(x["m"], x["src_wav"], g, so, dt, x["src_xyz"], x["rec_xyz"],
                                damp=x["damp"])
        resid = rec.detach() - x["obs"]
        gm, gq = torch.autograd.grad(rec, (x["m"], x["src_wav"]), grad_outputs=resid)
        return rec.detach(), gm, gq
    eng, traces, slots = st["engine"], [], []
    for s, n in enumerate(x["nts"]):
        out = torch.empty((n, case["rec"]), dtype=torch.float32, device=x["m"].device)
        slots.append(eng.add_shot(n, x["src_xyz"][s], st["wavs"][s], x["rec_xyz"][s], out))
        traces.append(out)
    while any(eng.steps_left(s) > 0 for s in slots):
        eng.step(32)
    eng.sync()
    for s in slots:
        eng.release(s)
    return traces


def work(case):
    """Bytes: the model read once, and per time step what a step cannot do without: every
    live wavefield level and coefficient read once, the new level written once, traces."""
    points = case["nz"] * case["ny"] * case["nx"]
    steps, shots, r = case["nt"] - 1, case["shots"], case["so"] // 2
    lap = 6 * r + 2 + 3 * r + 6          # adds and multiplies of one acoustic update
    traces = shots * case["nt"] * case["rec"] * 4
    kind = case["kind"]
    if kind == "tti":
        # p, r at two levels in, one out; m, epsilon, delta, theta, phi
        b = points * steps * (24 * shots + 20)
        f = points * steps * shots * (2 * 3 * 2 * 2 * 2 * r + 40)
        b += points * 20 + (16 * points * shots if case["final"] else 0)
    elif kind == "gradient":
        # forward for the traces; forward again, adjoint for the gradient (both levels in, one
        # out) and the imaging condition; adjoint for the wavelets
        b = points * steps * (4 * (12 * shots + 4) + 12 * shots)
        f = points * steps * shots * (4 * lap + 6)
        b += points * 8 + 3 * traces
    else:
        half = case.get("storage") == "f16" or (case.get("storage") == "auto" and case["so"] <= 8)
        coef = 8 if case.get("mask") else 4
        b = points * steps * (12 * shots + coef) / (2 if half else 1)
        f = points * steps * shots * lap
        b += points * 4 + (8 * points * shots if case.get("final") else 0)
        if kind == "serve":  # shots run 0.6 to 1 of the steps, evenly spread
            share = 0.8 + 0.2 / shots
            b, f, traces = share * b, share * f, share * traces
    return {"bytes": float(b + traces), "flops": float(f)}


# ---------------------------------------------------------------- 64-bit restatement

def _second_weights(r):
    f = math.factorial
    w = [0.0] * (r + 1)
    for k in range(1, r + 1):
        w[k] = 2.0 * (-1) ** (k + 1) * f(r) ** 2 / (k * k * f(r - k) * f(r + k))
    w[0] = -2.0 * sum(w[1:])
    return w


def _first_taps(r, stagger):
    """{offset: weight} of the first derivative: central (0), half a node ahead (+1) or
    behind (-1)."""
    f = math.factorial
    if stagger == 0:
        c = {k: (-1) ** (k + 1) * f(r) ** 2 / (k * f(r - k) * f(r + k)) for k in range(1, r + 1)}
        return {**c, **{-k: -v for k, v in c.items()}}
    odd = math.prod(range(1, 2 * r, 2))
    a = {k: (-1) ** (k + 1) * odd ** 2
         / (4 ** (r - 1) * (2 * k - 1) ** 2 * f(r + k - 1) * f(r - k)) for k in range(1, r + 1)}
    if stagger > 0:
        return {**{k: v for k, v in a.items()}, **{1 - k: -v for k, v in a.items()}}
    return {**{k - 1: v for k, v in a.items()}, **{-k: -v for k, v in a.items()}}


def _add_shifted(acc, q, axis, d, w):
    """acc(i) += w q(i + d e_axis), zero outside the grid."""
    n = q.shape[axis]
    if abs(d) >= n:
        return
    if d >= 0:
        acc.narrow(axis, 0, n - d).add_(q.narrow(axis, d, n - d), alpha=w)
    else:
        acc.narrow(axis, -d, n + d).add_(q.narrow(axis, 0, n + d), alpha=w)


def _laplacian(u, w, out):
    torch.mul(u, 3.0 * w[0] / H ** 2, out=out)
    for axis in range(3):
        for k in range(1, len(w)):
            _add_shifted(out, u, axis, k, w[k] / H ** 2)
            _add_shifted(out, u, axis, -k, w[k] / H ** 2)
    return out


def _derivative(q, axis, taps):
    out = torch.zeros_like(q)
    for d, w in taps.items():
        _add_shifted(out, q, axis, d, w / H)
    return out


def _points(xyz, shape):
    """Flat corner indices [n][8] and trilinear weights [n][8] of sparse points."""
    s = xyz.double() / H
    n = torch.tensor([shape[2], shape[1], shape[0]], device=xyz.device)
    i = torch.minimum(s.floor().long(), n - 2)
    fr = s - i
    idx, wgt = [], []
    for c in range(8):
        o = [(c >> a) & 1 for a in range(3)]
        idx.append(((i[:, 2] + o[2]) * shape[1] + i[:, 1] + o[1]) * shape[2] + i[:, 0] + o[0])
        p = [fr[:, a] if o[a] else 1.0 - fr[:, a] for a in range(3)]
        wgt.append(p[0] * p[1] * p[2])
    return torch.stack(idx, 1), torch.stack(wgt, 1)


def _damping(case, x):
    if case.get("mask"):
        return x["damp"].double()
    d = x["damp"].double()
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    return d[:nx][None, None, :] + d[nx:nx + ny][None, :, None] + d[nx + ny:][:, None, None]


def _sample(u, pts):
    return (u.reshape(-1)[pts[0]] * pts[1]).sum(1)


def _inject(u, b, pts, q):
    u.view(-1).index_add_(0, pts[0].reshape(-1),
                          (pts[1] * b.reshape(-1)[pts[0]] * q[:, None]).reshape(-1))


class _Acoustic:
    """The damped leapfrog of one shot in 64 bits."""

    def __init__(self, case, x, dt):
        self.shape = (case["nz"], case["ny"], case["nx"])
        damp = _damping(case, x)
        self.b = dt * dt / (x["m"].detach().double() + 0.5 * dt * damp)
        self.keep = 1.0 - damp * self.b / dt
        self.w = _second_weights(case["so"] // 2)
        self.lap = torch.empty_like(self.b)
        self.old = torch.zeros_like(self.b)
        self.now = torch.zeros_like(self.b)

    def step(self):
        """u- becomes u+ (sources not added yet)."""
        _laplacian(self.now, self.w, self.lap)
        self.old.sub_(self.now).mul_(-1.0).mul_(self.keep).add_(self.now)
        self.old.addcmul_(self.b, self.lap)
        self.old, self.now = self.now, self.old


def _exact_forward(case, x, dt, shot, nt, history=None):
    a = _Acoustic(case, x, dt)
    src, rec = _points(x["src_xyz"][shot], a.shape), _points(x["rec_xyz"][shot], a.shape)
    wav = x["src_wav"].detach()[shot].double()
    traces = torch.empty((nt, case["rec"]), device=wav.device, dtype=torch.float64)
    for n in range(nt):
        traces[n] = _sample(a.now, rec)
        if history is not None:
            history[n] = a.now
        if n < nt - 1:
            a.step()
            _inject(a.now, a.b, src, wav[n])
    return traces, a


def _exact_adjoint(case, x, dt, shot, resid, history=None, grad=None):
    """Wavelet gradient of a shot; with the forward history also adds to the model's."""
    nt = case["nt"]
    a = _Acoustic(case, x, dt)
    src, rec = _points(x["src_xyz"][shot], a.shape), _points(x["rec_xyz"][shot], a.shape)
    out = torch.zeros((nt, case["nsrc"]), device=resid.device, dtype=torch.float64)
    for n in range(nt - 1, 0, -1):
        if n < nt - 1:
            a.step()
        _inject(a.now, a.b, rec, resid[n])       # w^n = b lambda^n
        out[n - 1] = _sample(a.now, src)
        if grad is not None:
            d = history[n] - 2.0 * history[n - 1]
            if n >= 2:
                d += history[n - 2]
            grad.addcmul_(a.now, d, value=-1.0 / dt ** 2)
    return out


def _exact_tti(case, x, dt, shot):
    shape, r = (case["nz"], case["ny"], case["nx"]), case["so"] // 2
    stag = case["deriv"] == "staggered"
    inner, outer = _first_taps(r, 1 if stag else 0), _first_taps(r, -1 if stag else 0)
    damp = _damping(case, x)
    b = dt * dt / (x["m"].double() + 0.5 * dt * damp)
    keep = 1.0 - damp * b / dt
    a, s = 1.0 + 2.0 * x["eps"].double(), torch.sqrt(1.0 + 2.0 * x["delta"].double())
    th, ph = x["theta"].double(), x["phi"].double()
    n = [th.sin() * ph.cos(), th.sin() * ph.sin(), th.cos()]       # x, y, z
    axes = (2, 1, 0)
    src, rec = _points(x["src_xyz"][shot], shape), _points(x["rec_xyz"][shot], shape)
    wav = x["src_wav"][shot].double()
    zero = lambda: torch.zeros(shape, device=b.device, dtype=torch.float64)  # noqa: E731
    p, po, q, qo = zero(), zero(), zero(), zero()
    traces = torch.empty((case["nt"], case["rec"]), device=b.device, dtype=torch.float64)
    for t in range(case["nt"]):
        traces[t] = _sample(p if case["receiver"] == "p" else 0.5 * (p + q), rec)
        if t == case["nt"] - 1:
            break
        hxy, hz = zero(), zero()
        for field, dst, rotated in ((p, hxy, False), (q, hz, True)):
            g = [_derivative(field, ax, inner) for ax in axes]
            h = n[0] * g[0] + n[1] * g[1] + n[2] * g[2]
            for i, ax in enumerate(axes):
                dst += _derivative(n[i] * h if rotated else g[i] - n[i] * h, ax, outer)
        po.sub_(p).mul_(-1.0).mul_(keep).add_(p).addcmul_(b, a * hxy + s * hz)
        qo.sub_(q).mul_(-1.0).mul_(keep).add_(q).addcmul_(b, s * hxy + hz)
        p, po, q, qo = po, p, qo, q
        _inject(p, b, src, wav[t])
        _inject(q, b, src, wav[t])
    return traces, torch.stack([p, po]), torch.stack([q, qo])


def exact(case, seed):
    x, dt = _inputs(case, seed)
    kind, shots, nt = case["kind"], case["shots"], case["nt"]
    with torch.no_grad():
        if kind == "forward":
            got = []
            for s in range(shots):
                traces, a = _exact_forward(case, x, dt, s, nt)
                got.append((traces, torch.stack([a.now, a.old]) if case["final"] else None))
            rec = torch.stack([g[0] for g in got])
            return rec, torch.stack([g[1] for g in got]) if case["final"] else None
        if kind == "tti":
            got = [_exact_tti(case, x, dt, s) for s in range(shots)]
            rec = torch.stack([g[0] for g in got])
            if not case["final"]:
                return rec, None, None
            return rec, torch.stack([g[1] for g in got]), torch.stack([g[2] for g in got])
        if kind == "adjoint":
            return torch.stack([_exact_adjoint(case, x, dt, s, x["obs"][s].double())
                                for s in range(shots)])
        if kind == "gradient":
            grad = torch.zeros(x["m"].shape, device=x["m"].device, dtype=torch.float64)
            recs, gq = [], []
            for s in range(shots):
                hist = torch.empty((nt,) + tuple(grad.shape), device=grad.device,
                                   dtype=torch.float64)
                rec, _ = _exact_forward(case, x, dt, s, nt, hist)
                gq.append(_exact_adjoint(case, x, dt, s, rec - x["obs"][s].double(), hist, grad))
                recs.append(rec)
            return torch.stack(recs), grad, torch.stack(gq)
        return [_exact_forward(case, x, dt, s, n)[0] for s, n in enumerate(x["nts"])]
