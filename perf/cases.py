"""Timed cases of the phase-space lattice: what users of the library have it do, end to end through
the Python binding (paper_1508_02899_gb300.lat), with a 64-bit statement of the same results.

A case names one of six kinds of call; `prepare` builds the context, `run` makes the call.

  line      one 1D lattice in an Ornstein-Uhlenbeck flow: noise up, n steps, moments back
  ensemble  many independent 1D lattices advanced together, upwind or flux-limited drag
  plane     one 2D lattice (FP64, FP32, FP16 or BF16 storage) in an evolving random-phase flow, or
            frozen in the tilted cellular flow, upwind or flux-limited drag
  learned   the coarse 2D lattice with the learned closure (BF16 network) in an evolving flow
  train     loss and gradient of a rollout of the learned closure (one training iteration)
  observe   coarse-grained density moments and S1 of an ensemble's state
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_1508_02899_gb300 import inputs as I
from paper_1508_02899_gb300 import lat

DEV = "cuda"
L = 2 * math.pi
KAPPA = 1e-3
MU = 2.0 / 3.0
MODES = 8
NV_ANY_1D = (9, 17, 21, 33, 49, 65)      # 21 and 49 have no compiled kernel of their own
NV_LIM_1D = (9, 17, 33, 65)
NV_2D = (9, 13, 17, 19, 21, 33)
WIDTHS = (1, 2, 4, 8, 16, 32, 64, 128)
SEPS = (0, 1, 2, 4, 8, 16, 32, 64)
PARAMS = os.path.join(os.path.dirname(os.path.abspath(lat.__file__)), "closure_params.npz")
TORCH = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}


def listed():
    return [
        # the paper's 1D set-up watched closely: a few steps, then the moments, over and over;
        # launches and host work count here
        dict(name="line_f32_256x33_watch", kind="line", dtype="f32", nx=256, nv=33, steps=10,
             st=1.0),
        # a whole 1D run of the same set-up in double precision (1000 steps)
        dict(name="line_f64_256x33_run", kind="line", dtype="f64", nx=256, nv=33, steps=1000,
             st=1.0),
        # the ensemble average over 4096 flow realisations: the library's main workload
        dict(name="ensemble_f32_4096x65", kind="ensemble", dtype="f32", scheme="upwind", n=4096,
             nv=65, sizes="pow2", steps=20),
        # a small exploratory ensemble of arbitrary, odd grid sizes
        dict(name="ensemble_f32_64x33_ragged", kind="ensemble", dtype="f32", scheme="upwind",
             n=64, nv=33, sizes="ragged", steps=50),
        # the ensemble with the paper's flux limiter
        dict(name="ensemble_koren_f32_1024x65", kind="ensemble", dtype="f32", scheme="koren",
             n=1024, nv=65, sizes="pow2", steps=10),
        # the 2D lattice of the plain FP32 form
        dict(name="plane_f32_512x33", kind="plane", dtype="f32", scheme="upwind", flow="modes",
             nx=512, ny=512, nv=33, steps=10, st=1.0),
        # double precision in 2D, the size at which the other storage forms are validated
        dict(name="plane_f64_128x33", kind="plane", dtype="f64", scheme="upwind", flow="modes",
             nx=128, ny=128, nv=33, steps=10, st=1.0),
        # 16-bit storage, four times the grid of the FP32 form
        dict(name="plane_f16_1024x33", kind="plane", dtype="f16", scheme="upwind", flow="modes",
             nx=1024, ny=1024, nv=33, steps=6, st=1.0),
        # the paper's 2D runs: flux-limited drag in the tilted cellular flow
        dict(name="plane_koren_f32_1024x19", kind="plane", dtype="f32", scheme="koren",
             flow="cellular", nx=1024, ny=1024, nv=19, steps=4, st=1.0),
        # the learned closure on its coarse lattice (half a fine step)
        dict(name="learned_2048x9", kind="learned", nx=2048, ny=2048, nv=9, steps=2),
        # one training iteration of the closure: a rollout of 16 coarse steps and its adjoint
        dict(name="train_256x9", kind="train", nx=256, ny=256, nv=9, steps=16),
        # the paper's observables of an ensemble snapshot
        dict(name="observe_f32_1024x65", kind="observe", dtype="f32", n=1024, nv=65,
             sizes="pow2"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["line", "ensemble", "ensemble", "plane", "plane", "plane", "learned",
                       "train", "observe"])
    if kind == "line":
        return dict(kind=kind, dtype=rng.choice(["f32", "f32", "f64"]), nx=_log(rng, 64, 4096),
                    nv=rng.choice(NV_ANY_1D), steps=_log(rng, 4, 400),
                    st=rng.choice([0.1, 1.0, 10.0]))
    if kind == "ensemble":
        scheme = rng.choice(["upwind", "upwind", "koren"])
        return dict(kind=kind, dtype=rng.choice(["f32", "f32", "f32", "f64"]), scheme=scheme,
                    n=_log(rng, 8, 512), nv=rng.choice(NV_LIM_1D if scheme == "koren"
                                                       else NV_ANY_1D),
                    sizes=rng.choice(["pow2", "ragged"]), steps=_log(rng, 1, 24))
    if kind == "plane":
        scheme = rng.choice(["upwind", "upwind", "upwind", "koren"])
        dtype = rng.choice(["f64", "f32"] if scheme == "koren" else ["f64", "f32", "f32", "f16",
                                                                     "bf16"])
        flow = rng.choice(["modes", "cellular"])
        top = 160 if dtype == "f64" else 640
        unit = rng.choice([1, 4, 8, 8])       # any size, or whole vectors of the copy pipelines
        nx = max(unit, _log(rng, 40, top) // unit * unit)
        ny = nx if flow == "cellular" else _log(rng, 40, top)
        return dict(kind=kind, dtype=dtype, scheme=scheme, flow=flow, nx=nx, ny=ny,
                    nv=rng.choice(NV_2D), steps=_log(rng, 1, 8), st=rng.choice([0.1, 1.0, 10.0]))
    if kind == "learned":
        unit = rng.choice([1, 4, 128])
        return dict(kind=kind, nx=max(unit, _log(rng, 64, 1024) // unit * unit),
                    ny=_log(rng, 64, 1024), nv=rng.choice([9, 9, 13]), steps=_log(rng, 1, 8))
    if kind == "train":
        n = _log(rng, 32, 256)
        return dict(kind=kind, nx=n, ny=n, nv=9, steps=rng.choice([4, 8, 16]))
    return dict(kind=kind, dtype=rng.choice(["f32", "f64"]), n=_log(rng, 8, 512),
                nv=rng.choice(NV_LIM_1D), sizes=rng.choice(["pow2", "ragged"]))


# ---- inputs: what the user's program has, from the seed alone -----------------------------------
def _ensemble_table(c):
    """Sizes and parameters of the instances, the same for every seed."""
    koren = c.get("scheme") == "koren"
    rng = np.random.default_rng(77)
    if c["kind"] == "line":
        nx, st = np.array([c["nx"]]), np.array([c["st"]])
    else:
        n = c["n"]
        nx = (rng.choice([1024, 2048, 4096, 8192], size=n) if c["sizes"] == "pow2"
              else rng.integers(200, 1500, size=n))
        st = np.array([(0.1, 1.0, 10.0)[i % 3] for i in range(n)])
    tau = st * L
    seen = {}
    for a, b in zip(nx, tau):
        if (a, b) not in seen:
            seen[(a, b)] = I.choose_dt(1, int(a), L, c["nv"], float(b), KAPPA,
                                       cfl_factor=1 + MU if koren else 1.0)
    return nx.astype(np.int64), tau, np.array([seen[(a, b)] for a, b in zip(nx, tau)])


def _state_1d(c, seed, nx, dt):
    """Gaussian in v (0.2 V_max), the density modulated at random in space; instances
    concatenated as [j][x]."""
    nv, J = c["nv"], (c["nv"] - 1) // 2
    gen = torch.Generator(device=DEV).manual_seed(seed)
    out = torch.empty(int(nx.sum()) * nv, dtype=TORCH[c["dtype"]], device=DEV)
    j = torch.arange(-J, J + 1, dtype=torch.float64, device=DEV)
    g = torch.exp(-0.5 * (j / (0.2 * J)) ** 2)
    g = g / g.sum()
    m = 1 + 0.5 * torch.rand(int(nx.sum()), generator=gen, dtype=torch.float64, device=DEV)
    off = x0 = 0
    for n, d in zip(nx.tolist(), dt.tolist()):
        dv = (L / n) / d
        out[off:off + nv * n].view(nv, n).copy_(g[:, None] * (m[x0:x0 + n] / (1.25 * L * dv)))
        off += nv * n
        x0 += n
    return out


def _flow_1d(c, seed, n_inst):
    return I.flow1d_inputs(seed + 1, c.get("steps", 1), nmodes=MODES, n_inst=n_inst)


def _plane_setup(c):
    nx, nv = c["nx"], c["nv"]
    koren = c.get("scheme") == "koren"
    f = 1 + MU if koren else 1.0
    if c["kind"] in ("learned", "train"):   # the 33^2 (nv = 9) lattice restricted: dt / 4
        tau, kappa = L, KAPPA
        dt = I.choose_dt(2, nx, L, 4 * (nv - 1) + 1, tau, kappa) / 4
    elif c["flow"] == "cellular":           # Sec. 4.1: St = 1 / (2 pi), max |u| = 0.5
        tau, kappa = 1.0, 8 * math.pi * 1e-3
        dt = I.choose_dt(2, nx, L, nv, tau, kappa, u_rms=0.1, cfl_factor=f)
    else:
        tau, kappa = c["st"] * L, KAPPA
        dt = I.choose_dt(2, nx, L, nv, tau, kappa, cfl_factor=f)
    return dict(tau=tau, kappa=kappa, dt=dt, dx=L / nx, dv=(L / nx) / dt)


def _state_2d(c, p, seed, width=0.2):
    nx, ny, nv = c["nx"], c["ny"], c["nv"]
    J = (nv - 1) // 2
    gen = torch.Generator(device=DEV).manual_seed(seed)
    j = torch.arange(-J, J + 1, dtype=torch.float64, device=DEV)
    g = torch.exp(-0.5 * (j / (width * J)) ** 2)
    g = g / g.sum()
    m = 1 + 0.5 * torch.rand(ny, nx, generator=gen, dtype=torch.float64, device=DEV)
    m /= m.sum() * (p["dx"] * p["dv"]) ** 2
    f = torch.empty(nv, nv, ny, nx, dtype=torch.float64 if c.get("dtype") == "f64"
                    else torch.float32, device=DEV)
    for k in range(nv):
        f[k].copy_((g[k] * g)[:, None, None] * m)
    return f


def _flow_2d(c, p, seed):
    return I.flow2d_inputs(seed + 1, c["steps"], c["nx"], c["ny"], p["dx"])


def _cellular(c, dtype):
    return torch.tensor(np.stack(I.cellular_flow(c["nx"], c["ny"], L, 1.0)), dtype=dtype,
                        device=DEV)


def _params():
    with np.load(PARAMS) as z:
        return np.asarray(z["params"], dtype=np.float32)


# ---- the calls ----------------------------------------------------------------------------------
def prepare(case, seed):
    c = case
    if c["kind"] in ("line", "ensemble", "observe"):
        nx, tau, dt = _ensemble_table(c)
        f0 = _state_1d(c, seed, nx, dt)
        fl = _flow_1d(c, seed, len(nx))
        if c["kind"] == "line":
            ctx = lat.Lattice(f0, d=1, nx=int(nx[0]), nv=c["nv"], L=L, tau_p=float(tau[0]),
                              kappa=KAPPA, dt=float(dt[0]))
            ctx.set_flow_modes_1d(fl.k, fl.amp0[0], fl.tau_f, fl.sigma)
        else:
            n = len(nx)
            ctx = lat.Ensemble(f0, nv=c["nv"], nx=nx, L=np.full(n, L), tau_p=tau,
                               kappa=np.full(n, KAPPA), dt=dt)
            if c.get("scheme") == "koren":
                ctx.set_scheme(lat.SCHEME_KOREN, MU)
            ctx.set_flow_modes(fl.k, fl.amp0, fl.tau_f, fl.sigma)
        return dict(c=c, ctx=ctx, noise=fl.noise)
    p = _plane_setup(c)
    f0 = _state_2d(c, p, seed, 0.3 if c["kind"] == "train" else 0.2)
    half = c.get("dtype") in ("f16", "bf16")
    buf = torch.zeros(f0.shape, dtype=TORCH[c["dtype"]], device=DEV) if half else f0
    ctx = lat.Lattice(buf, d=2, nx=c["nx"], ny=c["ny"], nv=c["nv"], L=L, tau_p=p["tau"],
                      kappa=p["kappa"], dt=p["dt"])
    s = dict(c=c, ctx=ctx, noise=None)
    if half:
        ctx.encode(f0)
    if c.get("scheme") == "koren":
        ctx.set_scheme(lat.SCHEME_KOREN, MU)
    if c.get("flow") == "cellular":
        ctx.set_flow_field(_cellular(c, torch.float64 if c["dtype"] == "f64" else torch.float32))
    else:
        fl = _flow_2d(c, p, seed)
        frozen = c["kind"] == "train"
        ctx.set_flow_modes_2d(fl.kvec, fl.a, fl.phi0, math.inf if frozen else fl.tau_f)
        s["noise"] = None if frozen else fl.noise
    if c["kind"] in ("learned", "train"):
        ctx.learn(_params(), 2)
    if c["kind"] == "train":
        s["target"] = _state_2d(c, p, seed + 2, 0.29)
    return s


def run(state):
    c, ctx = state["c"], state["ctx"]
    if c["kind"] == "observe":
        coarse = ctx.coarse_moment(WIDTHS)
        num, den = ctx.s1(SEPS)
        return dict(coarse=coarse, s1_num=num, s1_den=den)
    if c["kind"] == "train":
        loss, grad = ctx.learn_grad(c["steps"], state["target"], 0.3)
        return dict(loss=loss, grad=grad)
    if state["noise"] is not None:
        ctx.set_noise(state["noise"])
    if c["kind"] == "learned":
        ctx.step(c["steps"])
        return dict(f=ctx.state)
    if c["kind"] == "ensemble":
        ctx.step(c["steps"])
        _, _, _, _, glob = ctx.moments()
        return dict(f=ctx.state, globals=glob)
    if c["kind"] == "line":
        _, rho, mv, mv2, glob = ctx.step_moments(c["steps"])
    else:
        ctx.step(c["steps"])
        _, rho, mv, mv2, glob = ctx.moments()
    f = ctx.decode()[0] if c.get("dtype") in ("f16", "bf16") else ctx.state
    return dict(f=f, rho=rho, mean_v=mv, mean_v2=mv2, globals=glob)


def work(case):
    """Each input read once, each output written once; arithmetic of the scheme as stated in
    `exact` (one operation per addition, multiplication, minimum or maximum)."""
    c = case
    size = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}[c.get("dtype", "f32")]
    koren = c.get("scheme") == "koren"
    if c["kind"] in ("line", "ensemble", "observe"):
        nx = _ensemble_table(c)[0]
        cells, cols = int(nx.sum()) * c["nv"], int(nx.sum())
        if c["kind"] == "observe":
            out = len(nx) * (len(WIDTHS) + 2 * len(SEPS)) * 8
            return dict(bytes=cells * size + out, flops=cells * (1 + 8 * len(SEPS)))
        moments = cells * 5
        return dict(bytes=2 * cells * size + len(nx) * (16 * 8 * c["steps"] + 24)
                    + (24 * cols if c["kind"] == "line" else 0),
                    flops=c["steps"] * (cells * (60 if koren else 14) + cols * 32) + moments)
    nxy = c["nx"] * c["ny"]
    cells = nxy * c["nv"] ** 2
    if c["kind"] == "learned":
        return dict(bytes=8 * cells, flops=c["steps"] * cells * (10496 + 60))
    if c["kind"] == "train":
        return dict(bytes=8 * cells + 4 * 5378, flops=c["steps"] * cells * 3 * (10496 + 60))
    out = 4 * cells if size == 2 else 0
    return dict(bytes=2 * cells * size + out + 32 * nxy,
                flops=c["steps"] * cells * (110 if koren else 27) + 7 * cells)


# ---- the same results in 64 bits ----------------------------------------------------------------
def exact(case, seed):
    c = case
    with torch.no_grad():
        if c["kind"] == "observe":
            return _exact_observe(c, seed)
        if c["kind"] in ("line", "ensemble"):
            return _exact_1d(c, seed)
        if c["kind"] == "plane":
            return _exact_plane(c, seed)
        if c["kind"] == "learned":
            p = _plane_setup(c)
            f = _state_2d(c, p, seed).double()
            W = _weights(torch.float64)
            for u in _flow_fields(c, p, seed):
                f = _learned_step(f, u, W, p)
            return dict(f=f)
    return _exact_train(c, seed)


def _upwind(f, ca, dim):
    """Difference of the upwind drag fluxes along one velocity axis."""
    n = f.shape[dim]
    lo, hi = f.narrow(dim, 0, n - 1), f.narrow(dim, 1, n - 1)
    F = ca.clamp(min=0).narrow(dim, 0, n - 1) * lo + ca.clamp(max=0).narrow(dim, 1, n - 1) * hi
    return _divergence(F, f, dim)


def _divergence(F, f, dim):
    """F_{j+1/2} - F_{j-1/2} for the interior faces F, zero on the walls."""
    n = f.shape[dim]
    out = torch.zeros_like(f)
    out.narrow(dim, 0, n - 1).add_(F)
    out.narrow(dim, 1, n - 1).sub_(F)
    return out


def _diffusion(f, r, dim):
    n = f.shape[dim]
    return _divergence(r * (f.narrow(dim, 1, n - 1) - f.narrow(dim, 0, n - 1)), f, dim)


def _increment(up2, up, down):
    dp, dm = down - up, up - up2
    nz = dp != 0
    th = dm / torch.where(nz, dp, torch.ones_like(dp))
    psi = torch.minimum((1.0 / 3.0 + th / 6.0).clamp(max=1.0), MU * th).clamp(min=0.0)
    return torch.where(nz, psi * dp, torch.zeros_like(dp))


def _limited(f, ca, dim):
    """Flux difference of the limited split fluxes (cells beyond the walls count as empty)."""
    n = f.shape[dim]

    def padded(q):
        shp = list(q.shape)
        shp[dim] = 1
        z = q.new_zeros(shp)
        return torch.cat([z, q, z], dim)

    P, M = padded(ca.clamp(min=0) * f), padded(ca.clamp(max=0) * f)

    def at(q, k):
        return q.narrow(dim, k, n - 1)

    F = (at(P, 1) + _increment(at(P, 0), at(P, 1), at(P, 2))
         + at(M, 2) + _increment(at(M, 3), at(M, 2), at(M, 1)))
    return _divergence(F, f, dim)


def _groups(nx, dt, tau):
    """Instances with the same size and parameters."""
    seen = {}
    for i, key in enumerate(zip(nx.tolist(), dt.tolist(), tau.tolist())):
        seen.setdefault(key, []).append(i)
    return seen


def _exact_1d(c, seed):
    nx, tau, dt = _ensemble_table(c)
    f0 = _state_1d(c, seed, nx, dt)
    fl = _flow_1d(c, seed, len(nx))
    nv, J = c["nv"], (c["nv"] - 1) // 2
    off = np.concatenate([[0], np.cumsum(nx * nv)])
    xoff = np.concatenate([[0], np.cumsum(nx)])
    out = torch.empty(f0.numel(), dtype=torch.float64, device=DEV)
    per = torch.zeros(3, int(nx.sum()), dtype=torch.float64, device=DEV)
    glob = np.zeros((len(nx), 3))
    noise = torch.tensor(fl.noise, device=DEV)
    amp0 = torch.tensor(fl.amp0, device=DEV)
    k = torch.tensor(fl.k, dtype=torch.float64, device=DEV)
    jv = torch.arange(-J, J + 1, dtype=torch.float64, device=DEV)[None, :, None]
    for (n, d, tp), members in _groups(nx, dt, tau).items():
        dx = L / n
        dv, g = dx / d, d / tp
        r = KAPPA * d / dv ** 2
        th = 2 * math.pi * ((k[:, None] * torch.arange(n, device=DEV)) % n) / n
        basis = torch.cat([torch.cos(th), torch.sin(th)])
        e = math.exp(-d / fl.tau_f)
        s = fl.sigma * math.sqrt(1 - e * e)
        size = max(1, 2 ** 26 // (n * nv))
        for i0 in range(0, len(members), size):
            idx = members[i0:i0 + size]
            f = torch.stack([f0[off[i]:off[i + 1]].view(nv, n) for i in idx]).double()
            amp = amp0[idx]
            for q in range(c["steps"]):
                f = torch.stack([torch.roll(f[:, j], j - J, 1) for j in range(nv)], 1)
                ca = g * ((amp @ basis)[:, None, :] / dv - jv)
                if c.get("scheme") == "koren":
                    y = f - _limited(f, ca, 1)
                    f = 0.5 * (f + y - _limited(y, ca, 1))
                else:
                    f = f - _upwind(f, ca, 1)
                f = f + _diffusion(f, r, 1)
                amp = amp * e + s * noise[q][idx]
            s0, s1, s2 = f.sum(1), (f * (jv * dv)).sum(1), (f * (jv * dv) ** 2).sum(1)
            w = torch.stack([s0.sum(1), s1.sum(1), s2.sum(1)], 1) * dx * dv
            glob[idx] = w.cpu().numpy()
            for a, i in enumerate(idx):
                out[off[i]:off[i + 1]] = f[a].reshape(-1)
                per[0, xoff[i]:xoff[i + 1]] = s0[a] * dv
                per[1, xoff[i]:xoff[i + 1]] = s1[a] / s0[a]
                per[2, xoff[i]:xoff[i + 1]] = s2[a] / s0[a]
    if c["kind"] == "ensemble":
        return dict(f=out, globals=glob)
    return dict(f=out, rho=per[0], mean_v=per[1], mean_v2=per[2], globals=glob[0])


def _exact_observe(c, seed):
    nx, tau, dt = _ensemble_table(c)
    f0 = _state_1d(c, seed, nx, dt)
    nv = c["nv"]
    off = np.concatenate([[0], np.cumsum(nx * nv)])
    coarse = np.zeros((len(nx), len(WIDTHS)))
    num, den = np.zeros((len(nx), len(SEPS))), np.zeros((len(nx), len(SEPS)))
    j = torch.arange(nv, dtype=torch.float64, device=DEV)
    dist = (j[:, None] - j[None, :]).abs()
    for (n, d, _), members in _groups(nx, dt, tau).items():
        dx = L / n
        dv = dx / d
        size = max(1, 2 ** 26 // (n * nv))
        for i0 in range(0, len(members), size):
            idx = members[i0:i0 + size]
            f = torch.stack([f0[off[i]:off[i + 1]].view(nv, n) for i in idx]).double()
            rho = f.sum(1)
            two = torch.cat([rho, rho], 1)
            for q, w in enumerate(WIDTHS):
                win = two[:, :n + w - 1].unfold(1, w, 1).sum(2) * (dv * dx)
                coarse[idx, q] = (win ** 2).mean(1).cpu().numpy()
            spread = dist @ f
            for q, s in enumerate(SEPS):
                num[idx, q] = ((spread * torch.roll(f, -s, 2)).sum(1).mean(1) * dv ** 3
                               ).cpu().numpy()
                den[idx, q] = ((rho * torch.roll(rho, -s, 1)).mean(1) * dv ** 2).cpu().numpy()
    return dict(coarse=coarse, s1_num=num, s1_den=den)


def _flow_fields(c, p, seed):
    """(u_x, u_y) of every step."""
    if c.get("flow") == "cellular":
        for _ in range(c["steps"]):
            yield _cellular(c, torch.float64)
        return
    fl = _flow_2d(c, p, seed)
    nx, ny = c["nx"], c["ny"]
    kv = torch.tensor(fl.kvec, device=DEV)
    i, l = torch.arange(nx, device=DEV), torch.arange(ny, device=DEV)
    tx = 2 * math.pi * ((kv[:, :1] * i) % nx).double() / nx
    ty = 2 * math.pi * ((kv[:, 1:] * l) % ny).double() / ny
    a = torch.tensor(fl.a, device=DEV)
    cx = -a * (2 * math.pi * kv[:, 1] / (ny * p["dx"]))
    cy = a * (2 * math.pi * kv[:, 0] / (nx * p["dx"]))
    phi = torch.tensor(fl.phi0, device=DEV)
    frozen = c["kind"] == "train"
    for n in range(c["steps"]):
        sy, cyy = torch.sin(ty + phi[:, None]), torch.cos(ty + phi[:, None])
        sx, cxx = torch.sin(tx), torch.cos(tx)
        yield torch.stack([(w[:, None] * sy).T @ cxx + (w[:, None] * cyy).T @ sx
                           for w in (cx, cy)])
        if not frozen:
            phi = phi + math.sqrt(2 * p["dt"] / fl.tau_f) * torch.tensor(fl.noise[n], device=DEV)


def _stream_2d(f):
    nv = f.shape[0]
    J = (nv - 1) // 2
    return torch.stack([torch.stack([torch.roll(f[a, b], (a - J, b - J), (0, 1))
                                     for b in range(nv)]) for a in range(nv)])


def _courant(u, nv, p):
    J = (nv - 1) // 2
    j = torch.arange(-J, J + 1, dtype=torch.float64, device=DEV)
    g = p["dt"] / p["tau"]
    return (g * (u[0] / p["dv"] - j[None, :, None, None]),
            g * (u[1] / p["dv"] - j[:, None, None, None]))


def _exact_plane(c, seed):
    p = _plane_setup(c)
    nv, J = c["nv"], (c["nv"] - 1) // 2
    r = p["kappa"] * p["dt"] / p["dv"] ** 2
    f = _state_2d(c, p, seed).double()
    rows = max(1, 2 ** 25 // (nv * nv * c["nx"]))   # grid rows taken at a time (bounds memory)
    for u in _flow_fields(c, p, seed):
        src, f = f, torch.empty_like(f)
        for y0 in range(0, c["ny"], rows):
            y1 = min(c["ny"], y0 + rows)
            yy = torch.arange(y0, y1, device=DEV)
            q = torch.stack([torch.stack([torch.roll(src[a, b][(yy - (a - J)) % c["ny"]], b - J, 1)
                                          for b in range(nv)]) for a in range(nv)])
            cx, cy = _courant(u[:, y0:y1], nv, p)
            cx, cy = cx.expand(1, nv, -1, -1), cy.expand(nv, 1, -1, -1)
            if c["scheme"] == "koren":
                y = q - _limited(q, cx, 1) - _limited(q, cy, 0)
                q = 0.5 * (q + y - _limited(y, cx, 1) - _limited(y, cy, 0))
            else:
                q = q - _upwind(q, cx, 1) - _upwind(q, cy, 0)
            f[:, :, y0:y1] = q + _diffusion(q, r, 1) + _diffusion(q, r, 0)
    s = torch.zeros(4, c["ny"], c["nx"], dtype=torch.float64, device=DEV)
    for a in range(nv):
        for b in range(nv):
            vx, vy = (b - J) * p["dv"], (a - J) * p["dv"]
            for k, w in enumerate((1.0, vx, vy, vx * vx + vy * vy)):
                s[k] += w * f[a, b]
    glob = (s.sum((1, 2)) * (p["dx"] * p["dv"]) ** 2).cpu().numpy()
    return dict(f=f, rho=(s[0] * p["dv"] ** 2).reshape(-1),
                mean_v=torch.cat([(s[1] / s[0]).reshape(-1), (s[2] / s[0]).reshape(-1)]),
                mean_v2=(s[3] / s[0]).reshape(-1), globals=glob)


def _weights(dtype):
    P = torch.tensor(_params(), dtype=dtype, device=DEV)
    at, out = 0, []
    for shp in ((16, 64), (64,), (64, 64), (64,), (64, 2), (2,)):
        n = int(np.prod(shp))
        out.append(P[at:at + n].view(shp))
        at += n
    return out


def _network(fs, inv, grads, cx, cy, g, *W):
    """Correction fluxes (interior vx and vy faces) of streamed rows fs [jy, jx, y, x]."""
    nv = fs.shape[0]
    pad = torch.nn.functional.pad(fs.permute(2, 3, 0, 1), (1, 1, 1, 1))
    X = [pad[..., a:a + nv, b:b + nv] * inv[..., None, None] for a in range(3) for b in range(3)]
    shape = X[0].shape
    X += [q[..., None, None].expand(shape) for q in grads]
    cax, cay = cx.permute(2, 3, 0, 1).expand(shape), cy.permute(2, 3, 0, 1).expand(shape)
    X = torch.stack(X + [cax, cay, torch.ones_like(cax)], -1)
    h = torch.relu(X @ W[0] + W[1])
    h = torch.relu(h @ W[2] + W[3])
    z = h @ W[4] + W[5]
    ca = (torch.stack([cax, cay], -1) - 0.5 * g).abs()
    b = torch.where(z > 0, 0.9 * (ca * (1 - ca)).clamp(min=0) * 0.5, torch.full_like(z, 0.25))
    y = (b * torch.tanh(z)).permute(4, 2, 3, 0, 1)
    return (y[0][:, :-1] * (fs[:, 1:] - fs[:, :-1]), y[1][:-1] * (fs[1:] - fs[:-1]))


def _learned_step(f, u, W, p):
    nv = f.shape[0]
    g = p["dt"] / p["tau"]
    r = p["kappa"] * p["dt"] / p["dv"] ** 2
    h = p["dt"] / (2 * p["dx"])
    grads = [(torch.roll(u[q], -1, d) - torch.roll(u[q], 1, d)) * h for q in (0, 1) for d in (1, 0)]
    cx, cy = _courant(u, nv, p)
    fs = _stream_2d(f)
    inv = 1.0 / fs.sum((0, 1))
    rows = max(1, 2 ** 21 // (nv * nv * f.shape[3]))
    parts = []
    for y0 in range(0, f.shape[2], rows):
        s = slice(y0, y0 + rows)
        q = fs[:, :, s]
        args = (q, inv[s], [v[s] for v in grads], cx[:, :, s], cy[:, :, s], g, *W)
        if torch.is_grad_enabled():
            gx, gy = checkpoint(_network, *args, use_reentrant=False)
        else:
            gx, gy = _network(*args)
        d = q - _upwind(q, cx[:, :, s], 1) - _upwind(q, cy[:, :, s], 0)
        d = d - _divergence(gx, q, 1) - _divergence(gy, q, 0)
        parts.append(d + _diffusion(d, r, 1) + _diffusion(d, r, 0))
    return torch.cat(parts, 2)


def _exact_train(c, seed):
    p = _plane_setup(c)
    f = _state_2d(c, p, seed, 0.3).double()
    target = _state_2d(c, p, seed + 2, 0.29).double()
    W = [w.clone().requires_grad_(True) for w in _weights(torch.float64)]
    for u in _flow_fields(c, p, seed):
        f = checkpoint(_learned_step, f, u, W, p, use_reentrant=False)
    d = f - target
    loss = (d * d).mean() + 0.3 * (d.sum((0, 1)) ** 2).mean()
    grads = torch.autograd.grad(loss, W)
    return dict(loss=float(loss.detach()),
                grad=torch.cat([q.reshape(-1) for q in grads]).cpu().numpy())
