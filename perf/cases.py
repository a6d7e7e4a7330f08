"""The work a user of this library has it do, as cases that can be timed and checked.

A case is one call of the public Python binding: forward modelling, the extended-model
gradient, the extended objective (a line search's evaluation without a gradient), the
pseudo-Hessian, the consistency term, or an l-BFGS direction.  ``exact`` computes the same
outputs in 64 bits with torch alone (the discrete scheme written as whole-array operations,
its gradient by automatic differentiation).
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

import paper_2305_14130_gb300 as efwi
from paper_2305_14130_gb300.optim import LBFGS

MODES = {"strain": 0, "strain_rate": 1, "velocity": 2}
ETA = (1e-3, 2e-3, 1e-3)

_WAVE = dict(rec="strain", source="moment", windows=False, ckpt=0, ckpt_store="fp32", snap_store="fp32", npml=20)


def _wave(name, call, nx, nz, dx, ns, nt, nch, **kw):
    return {"name": name, "call": call, "nx": nx, "nz": nz, "dx": dx, "ns": ns, "nt": nt, "nch": nch, **{**_WAVE, **kw}}


def listed():
    return [
        # one shot on a small grid: a first look at a model, a unit of a sweep; latency counts
        _wave("model_200x100_1", "forward", 200, 100, 2.0, 1, 1000, 80),
        _wave("grad_200x100_1", "gradient", 200, 100, 2.0, 1, 1000, 80),
        # a few shots on a small layered grid (differentiation checks, teaching, prototyping)
        _wave("grad_128x128_4", "gradient", 128, 128, 2.0, 4, 600, 100),
        # observed data of a whole guided-wave survey
        _wave("model_1000x300_32", "forward", 1000, 300, 1.0, 32, 300, 500),
        # the guided-wave inversion's gradient with the default options (FP32, sqrt(nt) checkpoints)
        _wave("grad_1000x300_32", "gradient", 1000, 300, 1.0, 32, 256, 500),
        # the same with FP16 storage chosen by the plan, on a subset of the shots
        _wave("grad_1000x300_8_half", "gradient", 1000, 300, 1.0, 8, 500, 500, ckpt="auto", ckpt_store="fp16",
              snap_store="fp16"),
        # a large survey where every shot has its own cropped window, FP16 checkpoints
        _wave("grad_3000x800_windows_6", "gradient", 3000, 800, 0.75, 6, 240, 600, windows=True, ckpt_store="fp16"),
        # line-search evaluation with 2-C geophones and vector-force sources
        _wave("objective_2000x600_4", "objective", 2000, 600, 1.0, 4, 256, 500, rec="velocity", source="force"),
        # a shot group of the largest grid, FP16 storage
        _wave("grad_4000x1200_2", "gradient", 4000, 1200, 0.5, 2, 240, 1500, ckpt="auto", ckpt_store="fp16",
              snap_store="fp16"),
        # illumination preconditioner of the comparison method
        _wave("hessian_1000x300_8", "hessian", 1000, 300, 1.0, 8, 300, 0),
        # consistency term of one parameter field over every component of a large extended model
        {"name": "consistency_2000x600_64", "call": "consistency", "nx": 2000, "nz": 600, "dx": 1.0, "ns": 64},
        # l-BFGS direction over the packed (Vp, Vs, rho) of the guided-wave problem, 5 pairs
        {"name": "direction_29M_5", "call": "direction", "n": 3 * 32 * 300 * 1000, "pairs": 5},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["forward", "gradient", "gradient", "gradient", "objective", "hessian", "consistency", "direction"])
    if call == "direction":
        return {"call": call, "n": _log(rng, 20_000, 28_000_000), "pairs": rng.randint(1, 6)}
    if call == "consistency":
        nx, nz = _log(rng, 120, 3000), _log(rng, 90, 900)
        ns = max(2, min(96, _log(rng, 2, 96), 70_000_000 // (nx * nz)))
        return {"call": call, "nx": nx, "nz": nz, "dx": 1.0, "ns": ns}
    nx, nz = _log(rng, 110, 4000), _log(rng, 90, 1200)
    npml = rng.choice([20, 20, 20, 12, 30])
    cells = (nx + 2 * npml + 2) * (nz + 2 * npml + 2)
    ns = max(1, min(_log(rng, 1, 32), 11_000_000 // cells))
    cost = {"forward": 1.0, "objective": 1.0, "hessian": 1.5, "gradient": 3.5}[call]
    nt = max(180, min(_log(rng, 180, 1000), int(9e9 / cost / (cells * ns))))
    case = _wave("", call, nx, nz, rng.choice([0.5, 0.75, 1.0, 2.0]), ns, nt, 0 if call == "hessian" else
                 _log(rng, 10, 600), npml=npml)
    del case["name"]
    case["windows"] = rng.random() < 0.3 and nx >= 200
    if call != "hessian":
        case["rec"] = rng.choice(["strain", "strain", "strain_rate", "velocity"])
    case["source"] = rng.choice(["moment", "moment", "moment", "force"])
    if call == "gradient":
        case["ckpt"] = rng.choice([0, 0, "auto"])
        case["ckpt_store"] = rng.choice(["fp32", "fp32", "fp16", "bf16"])
        case["snap_store"] = rng.choice(["fp32", "fp32", "fp16"])
    return case


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _smooth(nz, nx, corr, g):
    """Gaussian-smoothed white noise scaled to max 1 (periodic)."""
    f = torch.randn((nz, nx), generator=g, device="cuda", dtype=torch.float32)
    kx = torch.fft.rfftfreq(nx, device="cuda")[None] * corr
    kz = torch.fft.fftfreq(nz, device="cuda")[:, None] * corr
    f = torch.fft.irfft2(torch.fft.rfft2(f) * torch.exp(-2.0 * (math.pi ** 2) * (kx ** 2 + kz ** 2)), s=(nz, nx))
    return f / f.abs().max()


def _base_model(nx, nz, dx, g):
    """A 30 m low-velocity layer in faster rock with a +-3 % random field (FP32 on the device)."""
    z = torch.arange(nz, device="cuda", dtype=torch.float32) * dx
    mid = 0.5 * (nz - 1) * dx
    inside = ((z - mid).abs() < min(15.0, 0.2 * nz * dx))[:, None]
    corr = 20.0 / dx
    val = lambda a, b: torch.where(inside, torch.tensor(a, device="cuda"), torch.tensor(b, device="cuda")).expand(nz, nx)
    vp = val(3600.0, 4500.0) * (1 + 0.03 * _smooth(nz, nx, corr, g))
    vs = val(2000.0, 2600.0) * (1 + 0.03 * _smooth(nz, nx, corr, g))
    return [m.contiguous() for m in (vp, vs, val(2350.0, 2500.0))]


def _ricker(t, f0):
    a = (np.pi * f0 * t) ** 2
    return (1.0 - 2.0 * a) * np.exp(-a)


def _setup(case, seed):
    """Acquisition (host arrays), extended model and observed data (device FP32) of a case."""
    nx, nz, dx, ns, nt, nch = (case[k] for k in ("nx", "nz", "dx", "ns", "nt", "nch"))
    g, r = _gen(seed), np.random.default_rng(int(seed))
    base = _base_model(nx, nz, dx, g)
    # components of an inversion under way: the base model with a 1 % smooth update of their own
    model = []
    for m in base:
        upd = torch.stack([_smooth(nz, nx, 12.0, g) for _ in range(ns)])
        model.append((m[None] * (1 + 0.01 * upd)).contiguous())
    dt = 0.45 * dx / 4700.0
    f0 = 160.0 / dx
    width = (nx - 1) * dx
    win = None
    if case["windows"]:
        w = r.integers(max(80, nx // 5), max(100, 3 * nx // 5) + 1, ns)
        c = np.linspace(0.25, 0.75, ns) * nx
        x0 = np.clip((c - w // 2).astype(int), 0, nx - w)
        win = np.stack([x0, w], 1).astype(np.int32)
        xs = (x0 + 0.5 * w) * dx
    else:
        xs = width * (0.25 + 0.5 * (np.arange(ns) + 0.5) / ns)
    src = np.stack([xs + dx * r.uniform(-0.5, 0.5, ns), (0.5 * (nz - 1) + r.uniform(-1, 1, ns)) * dx], 1)
    amp = r.uniform(0.9, 1.1, ns)
    mt = 1e6 * np.stack([amp, 0.75 * amp, 0.2 * amp * r.uniform(-1, 1, ns)], 1)
    ang = r.uniform(0, 2 * np.pi, ns)
    force = 1e6 * np.stack([np.sin(ang), np.cos(ang)], 1) if case["source"] == "force" else None
    t = np.arange(nt + 1) * dt
    t0 = 1.5 / f0
    wav = np.stack([_ricker(t - t0 * r.uniform(0.95, 1.05), f0) for _ in range(ns)]).astype(np.float32)
    # a horizontal fibre (or a line of geophones) below the sources, where waves arrive within nt steps
    gauge = 10.0 * dx
    two = case["rec"] == "velocity"
    ptr, xz, tg = [0], [], []
    zf = (0.5 * (nz - 1) + max(5.0, min(0.13 * nz, 0.2 * (nt - 110))) + 0.3) * dx
    for s in range(ns):
        lo, wd = (0, nx) if win is None else win[s]
        cx = (lo + 8 + (wd - 17) * (np.arange(nch) + 0.5) / max(nch, 1)) * dx
        for tx, tz in (((1.0, 0.0), (0.0, 1.0)) if two else ((1.0, 0.0),)):
            xz.append(np.stack([cx, np.full(nch, zf)], 1))
            tg.append(np.tile([[tx, tz]], (nch, 1)))
        ptr.append(ptr[-1] + nch * (2 if two else 1))
    xz, tg = np.concatenate(xz), np.concatenate(tg)
    host = [m.cpu().numpy() for m in base]
    acq = SimpleNamespace(nx=nx, nz=nz, dx=dx, dz=dx, nt=nt, dt=dt, npml=case["npml"], pml_R=1e-3, pml_vmax=0.0,
                          pml_f0=f0, src_xz=src, mt=mt, wavelet=wav, tr_ptr=np.array(ptr, np.int32), ch_xz=xz, ch_t=tg,
                          gauge=gauge, das_mode=MODES[case["rec"]], win=win, force=force, ref_vp=host[0],
                          ref_vs=host[1], ref_rho=host[2])
    # observed traces: a direct arrival with the moveout of every channel, at the size of modelled data
    shot = np.repeat(np.arange(ns), np.diff(ptr))
    dist = np.hypot(xz[:, 0] - src[shot, 0], xz[:, 1] - src[shot, 1])
    k = 2 * np.pi * f0 / 4500.0
    size = 1e6 / (2500.0 * 4500.0 ** 2) * np.sqrt(k / (8 * np.pi))
    size *= {"strain": k, "strain_rate": k * k * 4500.0, "velocity": k * 4500.0}[case["rec"]]
    size *= 1.0 / k if force is not None else 1.0
    arr = torch.tensor(t0 + dist / 4500.0, device="cuda")[:, None]
    tt = torch.arange(1, nt + 1, device="cuda", dtype=torch.float64)[None] * dt - arr
    a = (math.pi * f0 * tt) ** 2
    d_obs = (1 - 2 * a) * torch.exp(-a) * torch.tensor(size / np.sqrt(dist + dx), device="cuda")[:, None]
    return acq, model, d_obs.float().contiguous(), src


def _zoi(ns, nx, nz, dx, seed):
    """One sinkhole per component along the middle of the grid, the outer taper at the sides."""
    r = np.random.default_rng(int(seed) + 7)
    x = (nx - 1) * dx * (0.2 + 0.6 * (np.arange(ns) + r.uniform(0, 1, ns)) / ns)
    return SimpleNamespace(active_x=np.tile([[0.15 * nx * dx, 0.85 * nx * dx]], (ns, 1)), taper=np.full(ns, 0.1 * nx * dx),
                           sink_xz=np.stack([x, np.full(ns, 0.5 * (nz - 1) * dx)], 1), sink_ax=np.full(ns, 12.0 * dx),
                           sink_az=np.full(ns, 6.0 * dx), n=2.0, nu=0.99)


def _field(case, seed):
    """One parameter field of an extended model under inversion, and the gradient it is added to."""
    nx, nz, ns = case["nx"], case["nz"], case["ns"]
    g = _gen(seed)
    base = _base_model(nx, nz, case["dx"], g)[0]
    m = torch.empty((ns, nz, nx), device="cuda")
    grad = torch.empty_like(m)
    for s in range(ns):
        m[s] = base * (1 + 0.01 * _smooth(nz, nx, 12.0, g))
        grad[s] = 1e-6 * _smooth(nz, nx, 6.0, g)
    return m, grad


def _pairs(case, seed):
    """A gradient and `pairs` curvature pairs (s, y), y = A s + a little noise, A > 0 diagonal."""
    n, g = case["n"], _gen(seed)
    rnd = lambda: torch.randn(n, generator=g, device="cuda")
    curv = torch.exp(rnd())
    ss = [rnd() for _ in range(case["pairs"])]
    ys = [curv * s + 0.02 * rnd() for s in ss]
    return rnd(), ss, ys


def prepare(case, seed):
    call = case["call"]
    if call == "direction":
        grad, ss, ys = _pairs(case, seed)
        opt = LBFGS(case["n"], m=max(case["pairs"], 1))
        for s, y in zip(ss, ys):
            opt.push(s, y)
        return SimpleNamespace(call=call, opt=opt, grad=grad)
    if call == "consistency":
        m, grad = _field(case, seed)
        nx, nz, ns, dx = case["nx"], case["nz"], case["ns"], case["dx"]
        b, bp, sink = efwi.zoi_weights(ns, nx, nz, dx, dx, _zoi(ns, nx, nz, dx, seed))
        # a shot group's plan: the term takes every component of the extended problem
        one = dict(case, ns=1, nt=4, nch=0, rec="strain", source="moment", windows=False, npml=20)
        plan = efwi.Plan(_setup(one, seed)[0], stencil="tma_pairs", tile=(32, 16), adj_tile=(32, 16),
                         adj_stencil="tma", overlap="off")
        return SimpleNamespace(call=call, plan=plan, m=m, g0=grad, w=(b, bp, sink))
    acq, model, d_obs, _ = _setup(case, seed)
    plan = efwi.Plan(acq, ckpt_interval=case["ckpt"], ckpt_store=case["ckpt_store"], snap_store=case["snap_store"])
    st = SimpleNamespace(call=call, plan=plan, model=model, d_obs=d_obs)
    if call == "objective":
        plan.set_zoi(_zoi(case["ns"], case["nx"], case["nz"], case["dx"], seed))
    return st


def run(st):
    if st.call == "forward":
        return st.plan.forward(*st.model)
    if st.call == "gradient":
        return st.plan.gradient(*st.model, st.d_obs)
    if st.call == "objective":
        return st.plan.extended_objective(*st.model, st.d_obs, ETA, None, None, None)
    if st.call == "hessian":
        return st.plan.pseudo_hessian(*st.model, eps=0.02)
    if st.call == "consistency":
        # the term is added to the data term's gradient
        return st.plan.regularization_grad(st.m, *st.w, 1e-3, g=st.g0.clone())
    return st.opt.direction(st.grad)


def _padded(case):
    p = 2 * (case["npml"] + 1)
    w = 0.4 * case["nx"] if case["windows"] else case["nx"]
    return case["ns"] * (w + p) * (case["nz"] + p)


def work(case):
    """One pass over the fields for every time step (no time step can start before the one before it
    has ended): 5 wavefields read and written and 5 materials read by a forward step (60 B a padded
    cell), 5 + 5 + 5 read, 5 + 5 written and the two forward velocities handed over by an adjoint
    step (116 B, or 108 B with 2-byte snapshots); the inputs and outputs once."""
    call = case["call"]
    if call == "direction":
        # g and every pair read, d written; a dot and an axpy for every vector
        return {"bytes": 4.0 * case["n"] * (2 + 2 * case["pairs"]), "flops": 8.0 * case["n"] * case["pairs"]}
    if call == "consistency":
        # m, b, b' (FP32) and the sinkhole flag read, the gradient read and written
        n = case["ns"] * case["nx"] * case["nz"]
        return {"bytes": 21.0 * n, "flops": 15.0 * n}
    cells, nt = _padded(case), case["nt"]
    phys = case["ns"] * case["nx"] * case["nz"]
    traces = case["ns"] * case["nch"] * (2 if case["rec"] == "velocity" else 1)
    data = 4.0 * traces * nt
    if call == "gradient":
        hand = 4 * 2 if case["snap_store"] == "fp32" else 2 * 2
        return {"bytes": cells * nt * (60.0 + 100 + 2 * hand) + 24.0 * phys + data, "flops": cells * nt * 190.0}
    more = {"forward": data, "objective": data + 27.0 * phys, "hessian": 8.0 * phys / case["ns"]}[call]
    return {"bytes": cells * nt * 60.0 + 12.0 * phys + more, "flops": cells * nt * 70.0}


# ---------------------------------------------------------------------------
# The same outputs in 64 bits, with torch alone
# ---------------------------------------------------------------------------

def _d(f, dim, fwd, h):
    """4th-order staggered difference along dim: to i + 1/2 (fwd) or from the half points to i."""
    n = f.shape[dim]
    pad = (2, 2) if dim == -1 else (0, 0, 2, 2)
    g = torch.nn.functional.pad(f, pad)
    at = lambda k: g.narrow(dim, 2 + k, n)
    if fwd:
        return (9 / 8 * (at(1) - at(0)) - 1 / 24 * (at(2) - at(-1))) / h
    return (9 / 8 * (at(0) - at(-1)) - 1 / 24 * (at(1) - at(-2))) / h


def _profile(n, p, h, npml, vmax, f0, dt, half):
    pos = torch.arange(n, dtype=torch.float64, device="cuda") + (0.5 if half else 0.0)
    dist = torch.clamp(torch.maximum((p - 1) - pos, pos - (n - p)), min=0.0)
    r = torch.clamp(dist / npml, max=1.0)
    d = -3.0 * vmax * math.log(1e-3) / (2.0 * npml * h) * r ** 2
    al = math.pi * f0 * (1 - r)
    b = torch.exp(-(d + al) * dt)
    return torch.where(d > 0, d * (b - 1) / torch.where(d > 0, d + al, torch.ones_like(d)), torch.zeros_like(d)), b


def _corners(x, z, ox, oz, h, x0, p, row):
    """Flat indices and bilinear weights [k, 4] of points on a sub-grid of the padded frame."""
    fi, fj = x / h - x0 + p - ox, z / h + p - oz
    i, j = np.floor(fi).astype(np.int64), np.floor(fj).astype(np.int64)
    ti, tj = fi - i, fj - j
    idx = np.stack([j * row + i, j * row + i + 1, (j + 1) * row + i, (j + 1) * row + i + 1], -1)
    w = np.stack([(1 - ti) * (1 - tj), ti * (1 - tj), (1 - ti) * tj, ti * tj], -1)
    return torch.tensor(idx, device="cuda"), torch.tensor(w, device="cuda", dtype=torch.float64)


class _Shots:
    """Time stepping of some shots with windows of one width, [k, NZ, NX] in float64."""

    def __init__(self, case, acq, shots):
        self.acq, self.shots = acq, shots
        p, h = case["npml"] + 1, acq.dx
        wins = [(0, acq.nx) if acq.win is None else tuple(int(v) for v in acq.win[s]) for s in shots]
        self.x0 = [w[0] for w in wins]
        self.w, self.p = wins[0][1], p
        self.NX, self.NZ = self.w + 2 * p, acq.nz + 2 * p
        vmax = float(acq.ref_vp.max())
        prof = lambda n, half: _profile(n, p, h, case["npml"], vmax, acq.pml_f0, acq.dt, half)
        X = lambda ab: [v[None, None, :] for v in ab]
        Z = lambda ab: [v[None, :, None] for v in ab]
        xi, xh, zi, zh = X(prof(self.NX, False)), X(prof(self.NX, True)), Z(prof(self.NZ, False)), Z(prof(self.NZ, True))
        self.pml = [xh, zi, xi, zh, xi, zi, zh, xh]
        self.wav = torch.tensor(acq.wavelet[shots], device="cuda", dtype=torch.float64)
        self.cell = acq.dx * acq.dz
        n = self.NX * self.NZ
        spread = {}
        for key, ox, oz in (("n", 0.0, 0.0), ("xz", 0.5, 0.5), ("vx", 0.5, 0.0), ("vz", 0.0, 0.5)):
            idx, w = zip(*[_corners(acq.src_xz[s:s + 1, 0], acq.src_xz[s:s + 1, 1], ox, oz, h, self.x0[k], p, self.NX)
                           for k, s in enumerate(shots)])
            idx = torch.cat([i + k * n for k, i in enumerate(idx)])
            spread[key] = (idx.reshape(-1), torch.cat(w))
        self.spread = spread
        f32 = lambda v: torch.tensor(np.asarray(v, np.float32).astype(np.float64), device="cuda")
        self.mt = f32(acq.mt[shots])
        self.force = None if acq.force is None else f32(acq.force[shots])
        # receivers: [traces, 4 components, 4 corners]
        rec_i, rec_w = [], []
        for k, s in enumerate(shots):
            a, b = int(acq.tr_ptr[s]), int(acq.tr_ptr[s + 1])
            c, t = acq.ch_xz[a:b], acq.ch_t[a:b]
            point = acq.das_mode == 2
            hl, sc = (0.0, 1.0) if point else (0.5 * acq.gauge, 1.0 / acq.gauge)
            ii, ww = [], []
            for sign in (1.0, -1.0):
                e = c + sign * hl * t
                for comp, ox, oz in ((0, 0.5, 0.0), (1, 0.0, 0.5)):
                    i, w = _corners(e[:, 0], e[:, 1], ox, oz, h, self.x0[k], p, self.NX)
                    keep = sc * (sign if not point else (1.0 if sign > 0 else 0.0))
                    ii.append(i + k * n)
                    ww.append(w * torch.tensor(t[:, comp:comp + 1] * keep, device="cuda"))
            rec_i.append(torch.stack(ii, 1))
            rec_w.append(torch.stack(ww, 1))
        self.rec_i, self.rec_w = torch.cat(rec_i), torch.cat(rec_w)

    def pad(self, m, ref):
        """Physical components in the frozen reference padding."""
        p, out = self.p, []
        ref = torch.tensor(ref, device="cuda", dtype=torch.float64)
        for k in range(len(self.shots)):
            a = torch.nn.functional.pad(ref[None, None, :, self.x0[k]:self.x0[k] + self.w], (p, p, p, p), mode="replicate")[0, 0]
            hole = torch.ones_like(a)
            hole[p:p + self.acq.nz, p:p + self.w] = 0
            out.append(a * hole + torch.nn.functional.pad(m[k, :, self.x0[k]:self.x0[k] + self.w], (p, p, p, p)))
        return torch.stack(out)

    def materials(self, vp, vs, rho):
        mu = rho * vs * vs
        lam = rho * (vp * vp - 2 * vs * vs)
        rep = lambda f: torch.nn.functional.pad(f[None], (0, 1, 0, 1), mode="replicate")[0]
        q, r = rep(1 / mu), rep(1 / rho)
        mxz = 4 / (q[:, :-1, :-1] + q[:, :-1, 1:] + q[:, 1:, :-1] + q[:, 1:, 1:])
        return lam, mu, mxz, 0.5 * (r[:, :-1, :-1] + r[:, :-1, 1:]), 0.5 * (r[:, :-1, :-1] + r[:, 1:, :-1])

    def zero(self):
        z = torch.zeros((len(self.shots), self.NZ, self.NX), dtype=torch.float64, device="cuda")
        return tuple(z for _ in range(13))

    def _inject(self, f, key, val):
        idx, w = self.spread[key]
        return f.reshape(-1).index_put((idx,), (w * val[:, None]).reshape(-1), accumulate=True).reshape(f.shape)

    def step(self, n, mats, st):
        """State and velocity samples [traces] after step n."""
        lam, mu, mxz, bx, bz = mats
        vx, vz, sxx, szz, sxz = st[:5]
        psi, h, dt, a = list(st[5:]), self.acq.dx, self.acq.dt, self.pml
        e = [_d(sxx, -1, True, h), _d(sxz, -2, False, h), _d(sxz, -1, False, h), _d(szz, -2, True, h)]
        for k in range(4):
            psi[k] = a[k][1] * psi[k] + a[k][0] * e[k]
        vx = vx + dt * bx * (e[0] + psi[0] + e[1] + psi[1])
        vz = vz + dt * bz * (e[2] + psi[2] + e[3] + psi[3])
        if self.force is not None:
            wn = self.wav[:, n] / self.cell * dt
            for key in ("vx", "vz"):
                b = (bx if key == "vx" else bz).reshape(-1)[self.spread[key][0]].reshape(-1, 4)
                idx, w = self.spread[key]
                val = (w * b * (wn * self.force[:, 0 if key == "vx" else 1])[:, None]).reshape(-1)
                if key == "vx":
                    vx = vx.reshape(-1).index_put((idx,), val, accumulate=True).reshape(vx.shape)
                else:
                    vz = vz.reshape(-1).index_put((idx,), val, accumulate=True).reshape(vz.shape)
        fx, fz = vx.reshape(-1), vz.reshape(-1)
        d = torch.zeros(self.rec_i.shape[0], dtype=torch.float64, device="cuda")
        for k in range(4):
            d = d + (self.rec_w[:, k] * (fx if k % 2 == 0 else fz)[self.rec_i[:, k]]).sum(-1)
        f = [_d(vx, -1, False, h), _d(vz, -2, False, h), _d(vx, -2, True, h), _d(vz, -1, True, h)]
        for k in range(4):
            psi[4 + k] = a[4 + k][1] * psi[4 + k] + a[4 + k][0] * f[k]
            f[k] = f[k] + psi[4 + k]
        tr = lam * (f[0] + f[1])
        sxx = sxx + dt * (tr + 2 * mu * f[0])
        szz = szz + dt * (tr + 2 * mu * f[1])
        sxz = sxz + dt * mxz * (f[2] + f[3])
        if self.force is None:
            dw = (self.wav[:, n + 1] - self.wav[:, n]) / self.cell
            sxx = self._inject(sxx, "n", -self.mt[:, 0] * dw)
            szz = self._inject(szz, "n", -self.mt[:, 1] * dw)
            sxz = self._inject(sxz, "xz", -self.mt[:, 2] * dw)
        return (vx, vz, sxx, szz, sxz, *psi), d

    def segment(self, n0, n1, mats, st):
        ds = []
        for n in range(n0, n1):
            st, d = self.step(n, mats, st)
            ds.append(d)
        return (torch.stack(ds, 1), *st)

    def data(self, rates):
        return self.acq.dt * torch.cumsum(rates, 1) if self.acq.das_mode == 0 else rates


def _groups(case, acq):
    """Shots that are stepped together: one window width, a bounded number of cells."""
    if acq.win is not None:
        return [[s] for s in range(acq.ns_)]
    cells = (acq.nx + 2 * case["npml"] + 2) * (acq.nz + 2 * case["npml"] + 2)
    k = max(1, 6_000_000 // cells)
    return [list(range(a, min(a + k, acq.ns_))) for a in range(0, acq.ns_, k)]


def _exact_wave(case, seed):
    acq, model, d_obs, _ = _setup(case, seed)
    acq.ns_ = case["ns"]
    nt, call = case["nt"], case["call"]
    grad = call == "gradient"
    m64 = [m.double() for m in model]
    ref = (acq.ref_vp, acq.ref_vs, acq.ref_rho)
    phi = torch.zeros((), dtype=torch.float64, device="cuda")
    data = torch.zeros((len(acq.ch_xz), nt), dtype=torch.float64, device="cuda")
    gs = [torch.zeros_like(m) for m in m64]
    hess = torch.zeros((acq.nz, acq.nx), dtype=torch.float64, device="cuda")
    for shots in _groups(case, acq):
        sh = _Shots(case, acq, shots)
        sub = [m[shots].requires_grad_(grad) for m in m64]
        a, b = int(acq.tr_ptr[shots[0]]), int(acq.tr_ptr[shots[-1] + 1])
        with torch.set_grad_enabled(grad):
            mats = sh.materials(*[sh.pad(m, r) for m, r in zip(sub, ref)])
            st, ds = sh.zero(), []
            if grad:
                k = max(1, int(math.sqrt(nt)))
                for n0 in range(0, nt, k):
                    out = checkpoint(sh.segment, n0, min(n0 + k, nt), mats, st, use_reentrant=False,
                                     preserve_rng_state=False)
                    ds.append(out[0])
                    st = out[1:]
                d = sh.data(torch.cat(ds, 1))
                part = 0.5 * ((d - d_obs[a:b].double()) ** 2).sum()
                for g, v in zip(gs, torch.autograd.grad(part, sub)):
                    g[shots] = v
                phi = phi + part.detach()
            else:
                p = sh.p
                for n in range(nt):
                    st, d = sh.step(n, mats, st)
                    ds.append(d)
                    if call == "hessian":
                        vx = 0.5 * (st[0][:, p:p + acq.nz, p - 1:p + sh.w - 1] + st[0][:, p:p + acq.nz, p:p + sh.w])
                        vz = 0.5 * (st[1][:, p - 1:p + acq.nz - 1, p:p + sh.w] + st[1][:, p:p + acq.nz, p:p + sh.w])
                        e = vx * vx + vz * vz
                        for q in range(len(shots)):
                            hess[:, sh.x0[q]:sh.x0[q] + sh.w] += e[q]
                data[a:b] = sh.data(torch.stack(ds, 1))
    if call == "forward":
        return data
    if grad:
        return (phi, *gs)
    if call == "hessian":
        c = 0.02 * hess.max()
        return hess, c / torch.clamp(hess, min=c)
    w = _exact_zoi(case, seed)
    reg = sum(_exact_reg(m, *w, e)[0] for m, e in zip(m64, ETA))
    return 0.5 * ((data - d_obs.double()) ** 2).sum(), reg


def _exact_zoi(case, seed):
    """Weights rounded to FP32 (they are inputs of the term) and sinkhole flags."""
    ns, nx, nz, dx = case["ns"], case["nx"], case["nz"], case["dx"]
    z = _zoi(ns, nx, nz, dx, seed)
    x = torch.arange(nx, device="cuda", dtype=torch.float64) * dx
    y = torch.arange(nz, device="cuda", dtype=torch.float64) * dx
    ln = math.log(z.nu)
    out = []
    for s in range(ns):
        far = torch.clamp(torch.maximum(z.active_x[s, 0] - x, x - z.active_x[s, 1]), min=0.0)
        dm = torch.sqrt((((x - z.sink_xz[s, 0]) / z.sink_ax[s]) ** 2)[None] + (((y - z.sink_xz[s, 1]) / z.sink_az[s]) ** 2)[:, None])
        f = lambda r: (torch.cos(0.5 * math.pi * torch.clamp(r, 0, 1)) ** z.n - ln) / (1 - ln)
        b = torch.minimum(f(far / z.taper[s])[None].expand(nz, nx), f(1 - dm))
        out.append((b, dm < 1))
    b = torch.stack([o[0] for o in out]).float().double()
    sink = torch.stack([o[1] for o in out])
    return b, torch.where(sink, torch.ones_like(b), b), sink


def _exact_reg(m, b, bp, sink, eta):
    """1/2 eta^2 |(I - S^T S_w) W m|^2 and its gradient, by slabs of rows (pixels are independent)."""
    phi, g = torch.zeros((), dtype=torch.float64, device="cuda"), torch.empty_like(m)
    for r in range(0, m.shape[1], 64):
        mm, bb, bs, sk = (v[:, r:r + 64] for v in (m, b, bp, sink))
        B, BM = bb.sum(0), (bb * mm).sum(0)
        one = torch.ones_like(bb)
        c = torch.where(sk & (m.shape[0] > 1), (1 - bb) / torch.where(sk, B - bb, one), torch.zeros_like(bb))
        dc = torch.where(sk & (m.shape[0] > 1), bb, one) - c * bb
        wm = dc * mm + c * BM
        om = bs / bs.sum(0)
        res = wm - (om * wm).sum(0)
        y = res - om * res.sum(0)
        phi = phi + 0.5 * eta * eta * (res ** 2).sum()
        g[:, r:r + 64] = eta * eta * (dc * y + bb * (c * y).sum(0))
    return phi, g


def exact(case, seed):
    call = case["call"]
    if call == "direction":
        g, ss, ys = _pairs(case, seed)
        q, al = g.double(), []
        for s, y in zip(reversed(ss), reversed(ys)):
            a = (s.double() @ q) / (s.double() @ y.double())
            al.append(a)
            q = q - a * y.double()
        q = q * ((ss[-1].double() @ ys[-1].double()) / (ys[-1].double() @ ys[-1].double()))
        for s, y, a in zip(ss, ys, reversed(al)):
            q = q + (a - (y.double() @ q) / (s.double() @ y.double())) * s.double()
        return -q
    if call == "consistency":
        m, grad = _field(case, seed)
        phi, g = _exact_reg(m.double(), *_exact_zoi(case, seed), 1e-3)
        return phi, grad.double() + g
    return _exact_wave(case, seed)
