"""Workloads that stand for what users run, for timing the library and comparing its outputs.

Each case is one call (or one optimisation step, or one serving tick) through the public entry
points in ``paper_2311_14780_gb300``, on seeded synthetic inputs shaped like the reflection
experiment: rectangle objects per wavelength, orthogonal Zernike-aberrated Gaussian probe modes, a
jittered raster, Poisson counts.  The inputs are made with plain torch, so they do not depend on the
library; ``exact`` states the same results in 64 bits, also with plain torch.

The evaluation point lies near the truth (a reconstruction in progress), data fitted with a Poisson
likelihood carry the model's background (without it, the darkest pixels' gradients are as uncertain as
the rounding of a field near zero), and Adam's moments are those of a run in progress: at the first
step Adam moves every parameter by the sign of its gradient, which turns the last bit of a gradient
near zero into a whole step.  Losses are FP64 sums of FP32 terms and are handed on as FP32, the way a
log keeps them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2311_14780_gb300 import api
from paper_2311_14780_gb300.autograd import ptycho_loss
from paper_2311_14780_gb300.serve import Request, Server

Z, PIXEL, TILT, LAMBDA0 = 88e-3, 15e-6, math.radians(70.0), 17.30e-9   # the experiment's geometry
LR_O, LR_P, LR_SIGMA, LR_BG, LR_DELTA = 1e-3, 1e-3, 1e-3, 1e-3, 1e-3
LR_SERVE = 5e-5
STEPS_DONE = 200
SERVE_ITERATIONS = 1 << 30
THRESHOLDS = (4.0, 65535.0)        # noisy and saturated camera pixels
B1, B2, ADAM_EPS = float(np.float32(0.9)), float(np.float32(0.999)), float(np.float32(1e-8))

BASE = {"kind": "step", "F": 256, "L": 3, "M": 4, "J": 400, "step": 24, "loss": "poisson", "remap": True,
        "bg": False, "sigma": False, "frame_mask": False, "batch": 0, "odd": 0}


def _case(**kw):
    c = dict(BASE)
    c.update(kw)
    return c


def listed():
    return [
        # plain single-mode, single-wavelength ptychography on a small crop: latency and launches
        _case(name="step_64_m1", F=64, L=1, M=1, J=64, step=16, loss="amplitude", remap=False),
        # the smallest fields of the throughput sweep: the passes that do not grow with the modes
        _case(name="step_128_m1", F=128, L=1, M=1, J=400, step=14, bg=True),
        # many modes and wavelengths on small frames
        _case(name="step_128_m8_l5", F=128, L=5, M=8, J=400, step=14, bg=True),
        # predicted patterns only (simulation, validation) at the experiment's 2 harmonics x 6 modes
        # and 225 positions
        _case(name="forward_256_m6_l2", kind="forward", F=256, L=2, M=6, J=225, step=29, bg=True),
        # the multiplexed reconstruction differentiated by torch: loss and both gradients
        _case(name="autograd_256_m4_l3", kind="autograd", bg=True),
        # a random subset of the positions per update, power coefficients, a mask per frame, odd sizes
        _case(name="minibatch_256_m3_l2", kind="minibatch", L=2, M=3, J=225, step=29, loss="amplitude", sigma=True,
              bg=True, frame_mask=True, batch=61, odd=3),
        # scan positions, powers and background optimised with the object and the probes
        _case(name="correct_256_m4_l3", kind="correct", sigma=True, bg=True),
        # the chirp-z propagator, every wavelength on one object grid
        _case(name="czt_256_m4_l2", kind="czt", L=2, M=4, J=144, step=29, loss="amplitude"),
        # one large field per position
        _case(name="step_512_m1", F=512, L=1, M=1, J=400, step=58, bg=True),
        # the 200-million-parameter reconstruction: the largest
        _case(name="step_512_m10_l6", F=512, L=6, M=10, J=900, step=96, bg=True),
        # the tilt correction of a stack of camera patterns, once per data set
        _case(name="tilt_256", kind="tilt", L=1, M=1, J=400, remap=False),
        # one tick of a server that holds sites of several shapes
        _case(name="serve_mix", kind="serve", J=100, F=0, L=0, M=0, step=0,
              sites="128,3,5,180;256,2,6,121;256,3,4,100;512,1,2,100"),
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "step", "forward", "autograd", "minibatch", "correct", "czt", "tilt", "serve"])
    logint = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    if kind == "tilt":                 # any frame size, odd ones among them
        F = logint(100, 1500)
        return _case(kind=kind, F=F, L=1, M=1, J=logint(4, max(5, min(900, 60_000_000 // (F * F)))), remap=False)
    if kind == "serve":
        sites = []
        for _ in range(rng.randint(2, 5)):
            F = rng.choice([128, 256, 512])
            sites.append("%d,%d,%d,%d" % (F, rng.randint(1, 3 if F == 512 else 5), rng.randint(1, 4 if F == 512 else 8),
                                          logint(50, 100 if F == 512 else 300)))
        return _case(kind=kind, J=100, F=0, L=0, M=0, step=0, sites=";".join(sites))
    F = rng.choice([64, 128, 256, 512])
    L, M = rng.randint(1, 6), rng.randint(1, 10)
    most = (2 if kind in ("correct", "czt") else 4) * 1200 * 512 * 512 // (F * F * L * M)
    J = logint(20, max(24, min(900, most)))
    loss = rng.choice(["amplitude", "poisson", "poisson_gaussian"])
    step = max(2, round(F * rng.uniform(0.08, 0.19)))
    return _case(kind=kind, F=F, L=L, M=M, J=J, step=step, loss=loss, remap=rng.random() < 0.7,
                 bg=loss != "amplitude" or kind == "correct" or rng.random() < 0.5, sigma=kind == "correct" or rng.random() < 0.4,
                 frame_mask=rng.random() < 0.3, batch=rng.randint(5, J) if kind == "minibatch" else 0,
                 odd=rng.randint(0, 7))


# --------------------------------------------------------------------------------------------------
# inputs (plain torch, from the seed alone)
# --------------------------------------------------------------------------------------------------

def _smooth(g, h, w, sigma):
    """Uniform noise blurred by a Gaussian (cyclic), scaled to [0, 1]."""
    u = torch.rand((h, w), generator=g, device="cuda")
    ky, kx = torch.fft.fftfreq(h, device="cuda")[:, None], torch.fft.rfftfreq(w, device="cuda")[None, :]
    s = torch.fft.irfft2(torch.fft.rfft2(u) * torch.exp(-2 * (math.pi * sigma) ** 2 * (ky * ky + kx * kx)), s=(h, w))
    lo, hi = s.aminmax()
    return (s - lo) / (hi - lo)


def _zernike(F, coeff):
    """Sum of the first ten Zernike polynomials (Noll) on the disk of radius F/2."""
    x = (torch.arange(F, device="cuda", dtype=torch.float64) - F / 2) / (F / 2)
    y, x = x[:, None], x[None, :]
    r2 = x * x + y * y
    terms = [torch.ones_like(r2), 2 * x + 0 * y, 2 * y + 0 * x, math.sqrt(3) * (2 * r2 - 1), math.sqrt(6) * 2 * x * y,
             math.sqrt(6) * (x * x - y * y), math.sqrt(8) * (3 * r2 - 2) * y, math.sqrt(8) * (3 * r2 - 2) * x,
             math.sqrt(8) * (3 * x * x * y - y ** 3), math.sqrt(8) * (x ** 3 - 3 * x * y * y)]
    return sum(c * t for c, t in zip(coeff, terms)) * (r2 <= 1)


def _probes(rng, F, L, M, ratio, photons):
    """[L, M, F, F] complex128: orthogonal modes of halving power, the width falling with the wavelength."""
    x = torch.arange(F, device="cuda", dtype=torch.float64) - F / 2
    r2 = x[:, None] ** 2 + x[None, :] ** 2
    power = 0.5 ** np.arange(M)
    power /= power.sum()
    P = torch.empty((L, M, F, F), dtype=torch.complex128, device="cuda")
    for l in range(L):
        s = 3.0 * F / 8.0 / ratio[l] / 2.3548
        amp = torch.exp(-r2 / (2 * s * s))
        modes = []
        for m in range(M):
            v = amp * torch.exp(1j * _zernike(F, rng.normal(0.0, 0.5, 10)))
            for u in modes:
                v = v - u * (u.conj() * v).sum()
            modes.append(v / torch.sqrt((v.abs() ** 2).sum()))
            P[l, m] = modes[-1] * math.sqrt(power[m] * photons / L)
    return P


def _objects(rng, g, shapes, ratio):
    """Random rectangles (8-40 px, about 30 %) on a smooth background, the same pattern at every
    wavelength's pixel size."""
    h, w = shapes[0]
    n = max(1, int(0.36 * h * w / (24 * 24)))
    size = rng.integers(8, 41, (n, 2))
    corner = np.stack([rng.integers(0, h, n), rng.integers(0, w, n)], 1)
    s = _smooth(g, h, w, 3.0)
    out = []
    for k, r in enumerate(ratio):
        y0, x0 = np.round(corner / r).astype(np.int64).T
        y1, x1 = np.minimum(np.round((corner + size) / r).astype(np.int64), [h, w]).T
        idx = np.concatenate([y0 * (w + 1) + x0, y1 * (w + 1) + x1, y0 * (w + 1) + x1, y1 * (w + 1) + x0])
        val = np.concatenate([np.ones(2 * n, np.int32), -np.ones(2 * n, np.int32)])
        d = np.zeros((h + 1) * (w + 1), np.int32)
        np.add.at(d, idx, val)
        inside = torch.from_numpy(d.reshape(h + 1, w + 1)).cuda().cumsum(0).cumsum(1)[:h, :w] > 0
        o = torch.where(inside, torch.polar(torch.full_like(s, 0.9), torch.full_like(s, 0.4 / r)),
                        torch.polar(torch.full_like(s, 0.5), 0.2 * s))
        out.append(o)
    return out


def _taps(F):
    """The tilted-plane remap: top-left model tap of each camera pixel (-1: none), its two weights."""
    c, s = math.cos(TILT), math.sin(TILT)
    X = (np.arange(F) - F / 2.0)[None, :] * PIXEL
    Y = (np.arange(F) - F / 2.0)[:, None] * PIXEL
    R = np.sqrt(X * X + Y * Y + Z * Z)
    yh = ((Y * c + Z * s) / R - s) / (PIXEL / Z * c) + F / 2.0
    xh = (X / R) / (PIXEL / Z) + F / 2.0
    ok = (yh >= 0) & (yh < F - 1) & (xh >= 0) & (xh < F - 1)
    iy, ix = np.where(ok, np.floor(yh), 0), np.where(ok, np.floor(xh), 0)
    base = np.where(ok, iy * F + ix, 0).astype(np.int64)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    return dev(ok), dev(base), dev(np.where(ok, yh - iy, 0.0)), dev(np.where(ok, xh - ix, 0.0))


def _remap(I, taps, F):
    """Bilinear interpolation of model-grid patterns [..., F, F] at the camera pixels (0 outside)."""
    ok, base, wy, wx = taps
    wy, wx, f = wy.to(I.dtype), wx.to(I.dtype), I.reshape(-1, F * F)
    b = base.reshape(-1)
    at = lambda o: f[:, (b + o).clamp(max=F * F - 1)].reshape(-1, F, F)  # noqa: E731
    v = (1 - wy) * ((1 - wx) * at(0) + wx * at(1)) + wy * ((1 - wx) * at(F) + wx * at(F + 1))
    return torch.where(ok, v, torch.zeros_like(v))


def _remap_t(D, taps, F):
    """The transpose of _remap."""
    ok, base, wy, wx = taps
    D = torch.where(ok, D, torch.zeros_like(D))
    g = torch.zeros((D.shape[0], F * F + F + 2), dtype=D.dtype, device=D.device)
    for o, w in ((0, (1 - wy) * (1 - wx)), (1, (1 - wy) * wx), (F, wy * (1 - wx)), (F + 1, wy * wx)):
        g.index_add_(1, base.reshape(-1) + o, (D * w).reshape(D.shape[0], -1))
    return g[:, :F * F].reshape(-1, F, F)


def _zoom_matrix(F, zeta):
    c = torch.arange(F, device="cuda", dtype=torch.float64) - F // 2
    return torch.exp(-2j * math.pi * zeta * c[:, None] * c[None, :] / F)


def _propagate(psi, zoom):
    """Orthonormal centred 2D DFT of [n, L, M, F, F], or the zoom DFT with the matrices ``zoom``."""
    if zoom is None:
        return torch.fft.fftshift(torch.fft.fft2(psi, norm="ortho"), dim=(-2, -1))
    F = psi.shape[-1]
    return torch.stack([(zoom[l] @ psi[:, l] @ zoom[l].T) / F for l in range(psi.shape[1])], 1)


def _propagate_t(Psi, zoom):
    if zoom is None:
        return torch.fft.ifft2(torch.fft.ifftshift(Psi, dim=(-2, -1)), norm="ortho")
    F = Psi.shape[-1]
    return torch.stack([(zoom[l].conj().T @ Psi[:, l] @ zoom[l].conj()) / F for l in range(Psi.shape[1])], 1)


def _windows(objs, pos, js, F):
    """Object windows [n, L, F, F] of positions js."""
    return torch.stack([torch.stack([o[pos[l, j, 0]:pos[l, j, 0] + F, pos[l, j, 1]:pos[l, j, 1] + F]
                                     for l, o in enumerate(objs)]) for j in js])


def _ramp(delta, js, F):
    """Phase ramps [n, L, F, F] of the Fourier shift by delta[l][j]."""
    f = torch.fft.fftfreq(F, device="cuda", dtype=torch.float64)
    d = delta.double()[:, js].permute(1, 0, 2)
    return torch.exp(2j * math.pi * (f[:, None] * d[..., 0, None, None] + f[None, :] * d[..., 1, None, None]))


def _chunks(js, cost):
    n = max(1, int(192e6 // cost))
    return [js[i:i + n] for i in range(0, len(js), n)]


def _problem(c, seed):
    """Everything a reconstruction has in hand, as torch tensors on the GPU (single precision)."""
    F, L, M, J = c["F"], c["L"], c["M"], c["J"]
    rng = np.random.default_rng([seed, F, L, M, J])
    g = torch.Generator(device="cuda")
    g.manual_seed(int(rng.integers(1 << 62)))
    czt = c["kind"] == "czt"
    ratio = [1.0 + 0.05 * l for l in range(L)]
    grid = [1.0] * L if czt else ratio                # chirp-z: every wavelength on one object grid
    n = math.ceil(math.sqrt(J))
    side = -(-((n - 1) * c["step"] + F + 8) // 16) * 16
    shapes = [(side + c["odd"], side + (c["odd"] * 3) % 8)] * L
    base = np.stack(np.divmod(np.arange(J), n), 1) * c["step"] + 3
    pos1 = base + rng.integers(-2, 3, base.shape)
    pos = np.stack([np.floor(pos1 / r + 0.5) for r in grid]).astype(np.int32)
    photons = 1e4 if F == 64 else 1e5
    truth_O, truth_P = _objects(rng, g, shapes, grid), _probes(rng, F, L, M, ratio, photons)
    p = {"F": F, "L": L, "M": M, "J": J, "shapes": shapes, "pos": pos, "loss": c["loss"], "remap": c["remap"],
         "eps": 1e-9 * photons / (F * F), "read_var": 2.0 if c["loss"] == "poisson_gaussian" else 0.0,
         "zoom": [1.0 / r for r in ratio] if czt else None, "lambdas": [LAMBDA0 * r for r in ratio]}
    rand = lambda *s: torch.rand(s, generator=g, device="cuda")  # noqa: E731
    p["sigma"] = 0.9 + 0.2 * rand(J) if c["sigma"] else None
    p["bg"] = (photons / (F * F)) * (0.05 + 0.1 * rand(F, F)) if c["bg"] else None
    if c["frame_mask"]:                               # hot pixels and a beam stop that moves
        m = rand(J, F, F) > 0.02
        for j in range(J):
            y, x = rng.integers(0, F, 2)
            m[j, y:y + F // 16, x:x + F // 16] = False
        p["mask"] = m.to(torch.uint8)
    else:
        p["mask"] = None
    p["batch"] = rng.permutation(J)[:c["batch"]].astype(np.int32) if c["batch"] else None
    p["delta"] = 0.8 * rand(L, J, 2) - 0.4 if c["kind"] == "correct" else None
    # Poisson counts of the truth (single precision; chirp-z data use the zoom matrices)
    P32 = truth_P.to(torch.complex64)
    zoom = [_zoom_matrix(F, z).to(torch.complex64) for z in p["zoom"]] if czt else None
    taps = _taps(F) if c["remap"] else None
    I = torch.empty((J, F, F), device="cuda")
    for js in _chunks(list(range(J)), 8 * L * M * F * F):
        psi = P32[None] * _windows(truth_O, pos, js, F)[:, :, None]
        if p["sigma"] is not None:
            psi = psi * p["sigma"][js][:, None, None, None, None]
        Psi = torch.view_as_real(_propagate(psi, zoom))
        I[js[0]:js[-1] + 1] = Psi.square_().sum(-1).sum((1, 2))
    if p["bg"] is not None:
        I += p["bg"]
    if taps is not None:
        for js in _chunks(list(range(J)), 24 * F * F):
            I[js[0]:js[-1] + 1] = _remap(I[js[0]:js[-1] + 1], taps, F)
    p["Im"] = torch.poisson(I, generator=g)
    # a point near the truth
    objs = []
    for o in truth_O:
        s1, s2 = _smooth(g, *o.shape, 4.0) - 0.5, _smooth(g, *o.shape, 4.0) - 0.5
        objs.append((o * torch.polar(1 + 0.05 * s1, 0.05 * s2)).reshape(-1))
    p["O"] = torch.cat(objs)
    p["P"] = truth_P
    for l in range(L):
        p["P"][l] *= torch.exp(1j * _zernike(F, rng.normal(0.0, 0.05, 10)))
    p["P"] = p["P"].to(torch.complex64)
    if c["kind"] == "correct":                        # powers still to be found, a few per cent off
        p["sigma"] = p["sigma"] * (1 + 0.03 * torch.randn(J, generator=g, device="cuda"))
    p["g"] = g
    return p


def _moments(p, n):
    """First and second Adam moments of a run in progress, for n real parameters."""
    return (0.1 * torch.randn(n, generator=p["g"], device="cuda"), 0.5 + torch.rand(n, generator=p["g"], device="cuda"))


def _plan(p):
    return api.Plan(p["F"], p["L"], p["M"], p["J"], p["shapes"], p["pos"], loss=p["loss"], eps=p["eps"],
                    remap=p["remap"], z=Z, det_pixel=PIXEL, tilt_rad=TILT, lambdas=p["lambdas"],
                    read_noise_var=p["read_var"], zoom=p["zoom"])


def _adam(p, plan, correct):
    kw = dict(lr_sigma=LR_SIGMA, lr_bg=LR_BG, lr_delta=LR_DELTA) if correct else {}
    st = api.AdamState(plan, LR_O, LR_P, **kw)
    st.t = STEPS_DONE
    for name in ("O", "P") + (("_sigma", "_bg", "_delta") if correct else ()):
        m, v = getattr(st, "m" + name), getattr(st, "v" + name)
        m0, v0 = _moments(p, m.numel())
        m.copy_(m0)
        v.copy_(v0)
    return st


def _serve_problems(c, seed):
    out = []
    for k, s in enumerate(c["sites"].split(";")):
        F, L, M, J = (int(v) for v in s.split(","))
        out.append(_problem(_case(kind="step", F=F, L=L, M=M, J=J, step=round(0.1125 * F)), seed * 16 + k))
    return out


def _camera(c, seed):
    """Raw camera patterns: a bright specular peak over speckle, clipped at a 16-bit full well."""
    F, J = c["F"], c["J"]
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1009 + F)
    x = torch.arange(F, device="cuda") - F / 2
    r2 = x[:, None] ** 2 + x[None, :] ** 2
    halo = torch.exp(-torch.sqrt(r2) / (0.25 * F)) * 60.0
    peak = 3e5 * torch.exp(-r2 / 2.0)
    I = torch.empty((J, F, F), device="cuda").exponential_(generator=g).clamp_(max=30.0).mul_(halo).add_(peak)
    return torch.poisson(I, generator=g).clamp_(max=65535.0)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "tilt":
        return {"kind": kind, "cam": _camera(case, seed)}
    if kind == "serve":
        sv, reqs, slots = Server(150 << 30), [], []
        for k, p in enumerate(_serve_problems(case, seed)):
            r = Request("site%d" % k, 0.0, p["F"], p["L"], p["M"], p["J"], p["shapes"], p["pos"], p["O"], p["P"], p["Im"],
                        iterations=SERVE_ITERATIONS, loss=p["loss"], eps=p["eps"], remap=p["remap"], z=Z,
                        det_pixel=PIXEL, tilt_rad=TILT, lr_O=LR_SERVE, lr_P=LR_SERVE)
            reqs.append(r)
            slots.append(sv.admit(r))
        return {"kind": kind, "server": sv, "reqs": reqs, "slots": slots}
    p = _problem(case, seed)
    plan = _plan(p)
    s = {"kind": kind, "p": p, "plan": plan}
    if kind in ("step", "correct", "czt"):
        s["adam"] = _adam(p, plan, kind == "correct")
    if p["delta"] is not None:
        p["delta"] = p["delta"].contiguous()
        plan.set_offsets(p["delta"])
    if p["batch"] is not None:
        s["batch"] = torch.from_numpy(p["batch"]).cuda()
    if kind == "autograd":
        p["O"].requires_grad_(True)
        p["P"].requires_grad_(True)
    return s


# --------------------------------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------------------------------

def run(s):
    kind = s["kind"]
    if kind == "tilt":
        out, mask = api.tilt_correct(s["cam"], Z, PIXEL, TILT, *THRESHOLDS)
        return {"patterns": out, "mask": mask}
    if kind == "serve":
        sv = s["server"]
        sv.tick()
        losses = [sv.status(k)[1] for k in s["slots"]]     # the request loop reads every site's status each tick
        return {"O": [r.O for r in s["reqs"]], "P": [r.P for r in s["reqs"]], "loss": losses}
    p, plan = s["p"], s["plan"]
    if kind == "forward":
        return {"I": plan.forward(p["O"], p["P"], p["sigma"], p["bg"])}
    if kind == "autograd":
        loss = ptycho_loss(p["O"], p["P"], plan, p["Im"], p["sigma"], p["bg"], p["mask"])
        gO, gP = torch.autograd.grad(loss, (p["O"], p["P"]))
        return {"loss": loss.detach().float(), "gO": gO, "gP": gP}
    if kind == "minibatch":
        loss, gO, gP = plan.adjoint(p["O"], p["P"], p["Im"], p["sigma"], p["bg"], p["mask"], s["batch"])
        return {"loss": loss.float(), "gO": gO, "gP": gP}
    a = s["adam"]
    loss = plan.step(a, p["O"], p["P"], p["Im"], p["sigma"], p["bg"], p["mask"])
    out = {"loss": loss.float(), "O": p["O"], "P": p["P"], "mO": a.mO, "vO": a.vO, "mP": a.mP, "vP": a.vP}
    if kind == "correct":
        out.update(sigma=p["sigma"], bg=p["bg"], delta=p["delta"], m_sigma=a.m_sigma, m_bg=a.m_bg, m_delta=a.m_delta)
    return out


def _bytes_of(c):
    F, L, M, J = c["F"], c["L"], c["M"], c["J"]
    n = math.ceil(math.sqrt(J))
    side = -(-((n - 1) * c["step"] + F + 8) // 16) * 16
    O, P, frames = 8 * L * side * side, 8 * L * M * F * F, 4 * J * F * F
    used = frames * c["batch"] // J if c["batch"] else frames
    mask = used // 4 if c["frame_mask"] else 0
    if c["kind"] == "forward":
        return O + P + frames
    if c["kind"] in ("autograd", "minibatch"):
        return 2 * (O + P) + used + mask
    return 6 * (O + P) + frames + mask                # parameters and both moments, read and written


def work(c):
    """Each input read once and each output written once; 5 N log2 N operations per DFT of N points."""
    if c["kind"] == "tilt":
        n = c["J"] * c["F"] * c["F"]
        return {"bytes": 9 * n, "flops": 8 * n}
    if c["kind"] == "serve":
        total = {"bytes": 0, "flops": 0}
        for s in c["sites"].split(";"):
            F, L, M, J = (int(v) for v in s.split(","))
            w = work(_case(kind="step", F=F, L=L, M=M, J=J, step=round(0.1125 * F)))
            total = {k: total[k] + w[k] for k in total}
        return total
    F, J = c["F"], c["batch"] or c["J"]
    dft2 = 10 * F * F * math.log2(F)
    flops = J * c["L"] * c["M"] * dft2 * (1 if c["kind"] == "forward" else 2)
    if c["kind"] == "czt":                            # one zoom DFT of F points: two DFTs of 2 F points
        flops *= 4 * math.log2(2 * F) / math.log2(F)
    if c["kind"] == "correct":                        # the shift of every window and its adjoint
        flops += 4 * J * c["L"] * dft2
    return {"bytes": _bytes_of(c), "flops": int(flops)}


# --------------------------------------------------------------------------------------------------
# the same results in 64 bits
# --------------------------------------------------------------------------------------------------

def _loss_64(I, Im, p):
    """Per-pixel loss and dL/dI."""
    Ie, Ih = I + p["eps"], Im.double()
    if p["loss"] == "amplitude":
        return (Ie.sqrt() - Ih.sqrt()) ** 2, 1 - (Ih / Ie).sqrt()
    if p["loss"] == "poisson_gaussian":
        Ie, Ih = Ie + p["read_var"], (Ih + p["read_var"]).clamp(min=0)
    log = torch.where(Ih > 0, Ih * torch.log(Ie / torch.where(Ih > 0, Ih, torch.ones_like(Ih))), torch.zeros_like(Ih))
    return Ie - Ih - log, 1 - Ih / Ie


def _adjoint_64(p, grad=True):
    """Loss and gradients (grad), or the predicted patterns, in complex128."""
    F, L, M, J, pos = p["F"], p["L"], p["M"], p["J"], p["pos"]
    O, objs, off = p["O"].detach().to(torch.complex128), [], 0
    for h, w in p["shapes"]:
        objs.append(O[off:off + h * w].reshape(h, w))
        off += h * w
    P = p["P"].detach().to(torch.complex128)
    zoom = [_zoom_matrix(F, z) for z in p["zoom"]] if p["zoom"] else None
    taps = _taps(F) if p["remap"] else None
    js_all = list(range(J)) if p["batch"] is None else [int(j) for j in p["batch"]]
    out = {"loss": 0.0, "gO": [torch.zeros_like(o) for o in objs], "gP": torch.zeros_like(P),
           "gs": torch.zeros(J, dtype=torch.float64, device="cuda"), "gb": torch.zeros((F, F), dtype=torch.float64, device="cuda"),
           "gd": torch.zeros((L, J, 2), dtype=torch.float64, device="cuda"),
           "I": None if grad else torch.empty((J, F, F), dtype=torch.float64, device="cuda")}
    freq = torch.fft.fftfreq(F, device="cuda", dtype=torch.float64)
    for js in _chunks(js_all, 16 * L * M * F * F):
        win = _windows(objs, pos, js, F)
        if p["delta"] is not None:
            ramp = _ramp(p["delta"], js, F)
            Q = torch.fft.fft2(win) * ramp
            win = torch.fft.ifft2(Q)
        sig = torch.ones(len(js), dtype=torch.float64, device="cuda") if p["sigma"] is None else p["sigma"].double()[js]
        s = sig[:, None, None, None]
        Psi = _propagate(P[None] * (s * win)[:, :, None], zoom)
        fields = (Psi.real ** 2 + Psi.imag ** 2).sum((1, 2))
        model = fields if p["bg"] is None else fields + p["bg"].double()
        cam = model if taps is None else _remap(model, taps, F)
        if not grad:
            out["I"][js[0]:js[-1] + 1] = cam
            continue
        terms, D = _loss_64(cam, p["Im"][js], p)
        use = torch.ones_like(D, dtype=torch.bool) if taps is None else taps[0].expand_as(D)
        if p["mask"] is not None:
            use = use & (p["mask"][js] != 0)
        out["loss"] += float(torch.where(use, terms, torch.zeros_like(terms)).sum())
        D = torch.where(use, D, torch.zeros_like(D))
        G = D if taps is None else _remap_t(D, taps, F)
        out["gb"] += G.sum(0)
        out["gs"][js] = 2 * (G * fields).sum((1, 2)) / sig
        chi = _propagate_t(2 * G[:, None, None] * Psi, zoom)
        del Psi
        out["gP"] += ((s * win).conj()[:, :, None] * chi).sum(0)
        patch = s * (P.conj()[None] * chi).sum(2)
        if p["delta"] is not None:
            Gh = torch.fft.fft2(patch)
            for a, f in ((0, freq[:, None]), (1, freq[None, :])):
                out["gd"][:, js, a] = ((Gh.conj() * (2j * math.pi * f) * Q).real.sum((-2, -1)) / (F * F)).T
            patch = torch.fft.ifft2(Gh * ramp.conj())
        for i, j in enumerate(js):
            for l in range(L):
                y, x = int(pos[l, j, 0]), int(pos[l, j, 1])
                out["gO"][l][y:y + F, x:x + F] += patch[i, l]
    out["gO"] = torch.cat([o.reshape(-1) for o in out["gO"]])
    return out


def _adam_64(theta, grad, m, v, t, lr):
    """Adam on real parameters (complex ones as pairs); returns the parameters and moments."""
    x = theta.detach()
    x = torch.view_as_real(x).double() if x.is_complex() else x.double()
    gr = torch.view_as_real(grad) if grad.is_complex() else grad
    gr = gr.reshape(-1)
    m = B1 * m.double() + (1 - B1) * gr
    v = B2 * v.double() + (1 - B2) * gr * gr
    lr = float(np.float32(lr))
    new = x.reshape(-1) - lr * (m / (1 - B1 ** t)) / ((v / (1 - B2 ** t)).sqrt() + ADAM_EPS)
    new = new.reshape(x.shape)
    return (torch.view_as_complex(new) if theta.is_complex() else new), m, v


def _tilt_64(cam):
    """The patterns at the camera position of every model pixel (bilinear, thresholds on the taps)."""
    J, F, _ = cam.shape
    c, s = math.cos(TILT), math.sin(TILT)
    da = PIXEL / Z
    db = da * c
    b = ((np.arange(F) - 0.5 * F) * db)[:, None]
    a = ((np.arange(F) - 0.5 * F) * da)[None, :]
    u = b + s
    w2 = 1.0 - a * a - u * u
    w = np.sqrt(np.where(w2 > 0, w2, 0.0))
    dy, dz = u * c - w * s, u * s + w * c
    ok = (w2 > 0) & (dz > 0)
    dz = np.where(ok, dz, 1.0)
    y, x = (Z * dy / dz) / PIXEL + 0.5 * F, (Z * a / dz) / PIXEL + 0.5 * F
    ok &= (y >= 0) & (y < F - 1) & (x >= 0) & (x < F - 1)
    y, x = np.where(ok, y, 0.0), np.where(ok, x, 0.0)
    dev = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()  # noqa: E731
    base = dev((np.floor(y) * F + np.floor(x)).astype(np.int64)).reshape(-1)
    fy, fx, ok = dev(y - np.floor(y)), dev(x - np.floor(x)), dev(ok)
    out = torch.zeros((J, F, F), dtype=torch.float64, device="cuda")
    for j in range(J):
        flat = cam[j].double().reshape(-1)
        t = [flat[base + o].reshape(F, F) for o in (0, 1, F, F + 1)]
        keep = ok.clone()
        for v in t:
            keep &= (v >= THRESHOLDS[0]) & (v < THRESHOLDS[1])
        val = (1 - fy) * ((1 - fx) * t[0] + fx * t[1]) + fy * ((1 - fx) * t[2] + fx * t[3])
        out[j] = torch.where(keep, val, torch.zeros_like(val))
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "tilt":
        return {"patterns": _tilt_64(_camera(case, seed)), "mask": None}
    if kind == "serve":
        out = {"O": [], "P": [], "loss": []}
        for p in _serve_problems(case, seed):
            r = _adjoint_64(p)
            zero = torch.zeros((), dtype=torch.float64, device="cuda")
            out["O"].append(_adam_64(p["O"], r["gO"], zero, zero, 1, LR_SERVE)[0])
            out["P"].append(_adam_64(p["P"], r["gP"], zero, zero, 1, LR_SERVE)[0])
            out["loss"].append(torch.tensor(r["loss"], dtype=torch.float64))
        return out
    p = _problem(case, seed)
    r = _adjoint_64(p, grad=kind != "forward")
    if kind == "forward":
        return {"I": r["I"]}
    loss = torch.tensor([r["loss"]], dtype=torch.float64)
    if kind == "autograd":
        return {"loss": loss.reshape(()), "gO": r["gO"], "gP": r["gP"]}
    if kind == "minibatch":
        return {"loss": loss, "gO": r["gO"], "gP": r["gP"]}
    out, t = {"loss": loss}, STEPS_DONE + 1
    for name, grad, lr in (("O", r["gO"], LR_O), ("P", r["gP"], LR_P)):
        m, v = _moments(p, 2 * p[name].numel())
        out[name], out["m" + name], out["v" + name] = _adam_64(p[name], grad, m, v, t, lr)
    if kind == "correct":
        for name, grad, lr in (("sigma", r["gs"], LR_SIGMA), ("bg", r["gb"], LR_BG), ("delta", r["gd"], LR_DELTA)):
            m, v = _moments(p, p[name].numel())
            out[name], out["m_" + name], _ = _adam_64(p[name], grad, m, v, t, lr)
    return out
