"""Workloads of the LBM-LETKF framework as its users run them, for timing.

A case is a dict of plain values. ``prepare`` makes what a program has in hand
(contexts, device arrays, host observations), ``run`` makes one pass through
the public entry points of ``paper_2308_03972_gb300`` and returns the whole
result, ``exact`` gives the same result in binary64 from plain torch, and
``work`` the bytes and operations that the result needs.

Kinds of case:
  cycle        set the members' velocities, forecast, mean velocity read-out,
               observe, analyse, read the posterior state (one
               data-assimilation cycle of an OSSE or a restart)
  forecast     the ensemble forecast alone, without observations
  analysis     the analysis alone of a state handed over by the caller
               (another model's ensemble, or an off-line re-analysis)
  batch        one cycle of several uneven experiments through ``Batch``
               (captured CUDA graph)
  adjoint      windowed misfit and its gradient through ``torch.autograd``
  diagnostics  moments, mean velocity and energy spectrum of an ensemble
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_2308_03972_gb300 import adjoint, binding, inputs

TAU0, CS, MU, BETA = 0.55, 0.2, 5e-4 * 0.001232, 1.05
U_RMS = 0.05 / math.sqrt(3.0)   # rms Mach number 0.05
SIGMA = 0.1 * U_RMS             # 10% observation error
SIGMA_RHO = 1e-3
CX = (0, 1, -1, 0, 0, 1, -1, 1, -1)
CY = (0, 0, 0, 1, -1, 1, -1, -1, 1)
W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4

# Twelve uneven experiments (lattice, members, observation lattice side,
# localisation radius): the batched configuration of the benchmark.
TWELVE = ("128:16:8:16 128:32:16:16 128:64:8:16 128:128:8:16 256:16:16:32 256:32:8:32 "
          "256:64:8:32 256:128:16:16 512:16:32:32 512:32:16:64 512:64:8:64 512:128:32:16")


def listed():
    return [
        # The tiny OSSE of the parity tests: what a user starts with, and the
        # size where launches and latency are everything.
        _da("tiny_cycle_f64", "cycle", 32, 32, 8, "fp64", 4, 4, 8.0, steps=10),
        # A lattice that is no multiple of anything, an odd ensemble size,
        # density observed with the velocity.
        _da("ragged_cycle_rho", "cycle", 90, 61, 21, "mixed", 6, 5, 12.5, steps=7, rho=True),
        # Spin-up of the benchmark ensemble: forecast only.
        {"name": "forecast_f32", "kind": "forecast", "nx": 256, "ny": 256, "k": 64, "prec": "mixed", "steps": 100},
        # The benchmark cycle (256^2 x 64, 8 x 8 points) in both precisions.
        _da("cycle_f32", "cycle", 256, 256, 64, "mixed", 8, 8, 32.0, steps=10),
        _da("cycle_f64", "cycle", 256, 256, 64, "fp64", 8, 8, 32.0, steps=10),
        # Dense observations (the precision sweep's lattices): more local
        # scalars than members, so the local problem is as large as the
        # ensemble. Small, middle and large ensembles.
        _da("dense_k16", "analysis", 256, 256, 16, "mixed", 32, 32, 32.0),
        _da("dense_k32", "analysis", 256, 256, 32, "mixed", 16, 16, 32.0),
        _da("dense_k64", "analysis", 256, 256, 64, "mixed", 32, 32, 32.0),
        # A large ensemble with fewer local scalars than members, but more
        # than a warp holds.
        _da("wide_k128", "analysis", 128, 128, 128, "mixed", 16, 16, 16.0),
        # The twelve uneven experiments in one batch.
        {"name": "batch_twelve", "kind": "batch", "experiments": TWELVE, "steps": 10},
        # The adjoint configuration: 200-step window, 64 initial states.
        {"name": "adjoint_f32", "kind": "adjoint", "nx": 256, "ny": 256, "k": 64, "prec": "mixed", "nobs_x": 16,
         "nobs_y": 16, "steps": 200, "every": 10, "checkpoint": 20},
        # What an OSSE records of its ensemble.
        {"name": "diagnostics_f32", "kind": "diagnostics", "nx": 256, "ny": 256, "k": 64, "prec": "mixed"},
    ]


def _da(name, kind, nx, ny, k, prec, nobs_x, nobs_y, d_cut, steps=0, rho=False):
    c = {"kind": kind, "nx": nx, "ny": ny, "k": k, "prec": prec, "nobs_x": nobs_x, "nobs_y": nobs_y,
         "d_cut": float(d_cut), "steps": steps, "rho": rho}
    return dict(c, name=name) if name else c


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the listed kinds: lattices 24..320 per side, 4..128 members,
    observation spacings of 4..32 cells, d_cut of 0.6..4 spacings."""
    most = max(_effort(c) for c in listed())
    while True:
        c = _draw(rng)
        if _effort(c) <= most:
            return c


def _draw(rng):
    kind = rng.choice(["cycle", "cycle", "cycle", "forecast", "analysis", "analysis", "analysis", "batch", "adjoint",
                       "diagnostics"])
    if kind == "batch":
        side = [rng.choice([48, 64, 96, 128, 160, 192, 256]) for _ in range(rng.randint(2, 6))]
        ex = []
        for n in side:
            spacing = rng.choice([8, 16, 32])
            ex.append("%d:%d:%d:%g" % (n, rng.choice([8, 16, 24, 32, 48, 64, 128]), max(2, n // spacing),
                                       rng.choice([0.5, 1.0, 2.0]) * spacing))
        return {"kind": kind, "experiments": " ".join(ex), "steps": 2 * rng.randint(1, 10)}
    nx, ny, k = _log_int(rng, 24, 320), _log_int(rng, 24, 320), _log_int(rng, 4, 128)
    if rng.random() < 0.5:
        k = max(4, k // 4 * 4)
    prec = rng.choice(["mixed", "mixed", "mixed", "fp64"])
    if kind in ("cycle", "analysis"):
        if prec == "fp64":
            k = min(k, 64)
        spacing = _log_int(rng, 4, 32)
        return _da(None, kind, nx, ny, k, prec, min(64, max(2, nx // spacing)), min(64, max(2, ny // spacing)),
                   round(spacing * math.exp(rng.uniform(math.log(0.6), math.log(4.0))), 2),
                   steps=rng.randint(1, 20) if kind == "cycle" else 0, rho=rng.random() < 0.25)
    c = {"kind": kind, "nx": nx, "ny": ny, "k": k, "prec": prec}
    if kind == "forecast":
        c["steps"] = _log_int(rng, 1, 150)
    if kind == "adjoint":
        steps = _log_int(rng, 5, 200)
        c.update(nobs_x=max(2, nx // 16), nobs_y=max(2, ny // 16), steps=steps, every=rng.randint(1, min(20, steps)),
                 checkpoint=rng.randint(2, 25))
    return c


def _effort(c):
    """Rough cost on one scale, for keeping drawn cases below the listed ones."""
    if c["kind"] == "batch":
        return sum(_effort(dict(e, steps=c["steps"])) for e in _experiments(c))
    f64 = c["prec"] == "fp64"
    per = 24.0 if f64 else 1.0
    upd = c["nx"] * c["ny"] * c["k"]
    e = 72.0 * per * upd * c.get("steps", 0) * (5 if c["kind"] == "adjoint" else 1)
    if c["kind"] == "diagnostics":
        e += 8.0 * upd * (c["nx"] + c["ny"])
    if c["kind"] in ("cycle", "analysis"):
        area = math.pi * (2 * c["d_cut"] + 1) ** 2 / (c["nx"] * c["ny"])
        p = (3 if c["rho"] else 2) * math.ceil(min(1.0, area) * c["nobs_x"] * c["nobs_y"])
        n = min(c["k"], p + 4)
        e += 0.5 * per * ((3 if c["rho"] else 2) * c["nobs_x"] * c["nobs_y"]) ** 2 * c["k"]
        e += c["nx"] * c["ny"] * ((100.0 if f64 else 20.0) * n ** 3 + 4.0 * per * p * c["k"] ** 2 * (p >= c["k"]))
    return e


# ---- inputs ------------------------------------------------------------------

def _experiments(c):
    out = []
    for t in c["experiments"].split():
        n, k, no, dc = t.split(":")
        out.append({"kind": "cycle", "nx": int(n), "ny": int(n), "k": int(k), "prec": "mixed", "nobs_x": int(no),
                    "nobs_y": int(no), "d_cut": float(dc), "rho": False, "steps": c["steps"]})
    return out


def _velocity(nx, ny, count, gen):
    """count divergence-free random-phase velocity fields with E(k) ~ k^-3 for
    1 <= |k| <= min(nx, ny) / 4 and rms speed U_RMS: u, v [ny][nx][count]."""
    dev = "cuda"
    kx = torch.fft.fftfreq(nx, 1.0 / nx, dtype=torch.float64, device=dev)[None, :]
    ky = torch.fft.fftfreq(ny, 1.0 / ny, dtype=torch.float64, device=dev)[:, None]
    kk = torch.sqrt(kx * kx + ky * ky)
    band = (kk >= 1.0) & (kk <= max(2.0, min(nx, ny) / 4.0))
    amp = torch.where(band, torch.where(band, kk, torch.ones_like(kk)) ** -3.0, torch.zeros_like(kk))
    u = torch.empty((ny, nx, count), dtype=torch.float64, device=dev)
    v = torch.empty_like(u)
    for a in range(0, count, 32):
        b = min(count, a + 32)
        ph = torch.rand((b - a, ny, nx), dtype=torch.float64, device=dev, generator=gen) * (2.0 * math.pi)
        psi = torch.polar(amp.expand_as(ph), ph)
        uu = torch.fft.ifft2(1j * ky / ny * psi).real
        vv = torch.fft.ifft2(-1j * kx / nx * psi).real
        s = U_RMS / torch.sqrt((uu * uu + vv * vv).mean(dim=(1, 2), keepdim=True))
        u[:, :, a:b] = (uu * s).permute(1, 2, 0)
        v[:, :, a:b] = (vv * s).permute(1, 2, 0)
    return u, v


def _members(nx, ny, k, gen):
    """An ensemble: a common random field plus a tenth of a field per member."""
    uc, vc = _velocity(nx, ny, 1, gen)
    up, vp = _velocity(nx, ny, k, gen)
    return (uc + 0.1 * up).contiguous(), (vc + 0.1 * vp).contiguous()


def _observations(c, gen, times=1):
    """Points and noisy values [times][npts] of a random true flow (host arrays)."""
    ix, iy = inputs.uniform_obs_points(c["nx"], c["ny"], c["nobs_x"], c["nobs_y"])
    tu, tv = _velocity(c["nx"], c["ny"], 1, gen)
    at = (torch.as_tensor(iy, dtype=torch.long), torch.as_tensor(ix, dtype=torch.long))
    z = torch.randn((3, times, len(ix)), dtype=torch.float64, device="cuda", generator=gen).cpu().numpy()
    yu = tu[:, :, 0].cpu()[at].numpy() + SIGMA * z[0]
    yv = tv[:, :, 0].cpu()[at].numpy() + SIGMA * z[1]
    return ix, iy, yu, yv, 1.0 + SIGMA_RHO * z[2]


def _equilibrium(rho, u, v):
    uu = 1.5 * (u * u + v * v)
    f = torch.empty((9,) + tuple(u.shape), dtype=u.dtype, device=u.device)
    for a in range(9):
        cu = CX[a] * u + CY[a] * v
        f[a] = rho * W[a] * (1.0 + 3.0 * cu + 4.5 * cu * cu - uu)
    return f


def _inputs(c, seed, which=0):
    """Everything random about a case, from the seed alone."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1000003 * int(seed) + 7919 * which + 17)
    x = {"force": inputs.forcing_field(c["nx"], c["ny"], int(seed) % 100003, 3.5e-6)}
    x["u"], x["v"] = _members(c["nx"], c["ny"], c["k"], gen)
    if c["kind"] in ("analysis", "adjoint"):
        rho = 1.0 + 1e-3 / U_RMS * 0.1 * (x["u"] - x["u"].mean(dim=2, keepdim=True))
        x["f"] = _equilibrium(rho, x["u"], x["v"])
        del x["u"], x["v"]
    if c["kind"] in ("cycle", "analysis"):
        x["obs"] = tuple(o[0] if o.ndim == 2 else o for o in _observations(c, gen))
    if c["kind"] == "adjoint":
        x["obs"] = _observations(c, gen, c["steps"] // c["every"])
    return x


# ---- prepare / run -------------------------------------------------------------

def _ensemble(c, force):
    prec = binding.LBM_FP64 if c["prec"] == "fp64" else binding.LBM_MIXED
    return binding.Ensemble(c["nx"], c["ny"], c["k"], TAU0, CS, MU, prec, force=force)


def _out(c):
    return torch.empty((9, c["ny"], c["nx"], c["k"]), dtype=torch.float64, device="cuda")


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "batch":
        members = []
        for i, e in enumerate(_experiments(c)):
            x = _inputs(e, seed, i)
            members.append({"case": e, "x": x, "ens": _ensemble(e, x["force"]), "out": _out(e)})
        return {"case": c, "members": members, "batch": binding.Batch([m["ens"] for m in members])}
    s = {"case": c, "x": _inputs(c, seed)}
    s["ens"] = _ensemble(c, s["x"]["force"])
    if c["kind"] == "adjoint":
        ix, iy, yu, yv, _ = s["x"]["obs"]
        s["win"] = binding.Window(c["steps"], c["every"], ix, iy, yu, yv, SIGMA, SIGMA, c["checkpoint"])
        s["f0"] = s["x"]["f"].requires_grad_(True)
        s["cs"] = torch.tensor(CS, dtype=torch.float64, requires_grad=True)
        return s
    if c["kind"] == "diagnostics":
        shape = (c["ny"], c["nx"], c["k"])
        s["ens"].set_equilibrium(None, s["x"]["u"], s["x"]["v"])
        s["moments"] = [torch.empty(shape, dtype=torch.float64, device="cuda") for _ in range(3)]
        s["E"] = torch.empty(binding.spectrum_shells(c["nx"], c["ny"]), dtype=torch.float64, device="cuda")
    else:
        s["out"] = _out(c)
    s["mean"] = [torch.empty((c["ny"], c["nx"]), dtype=torch.float64, device="cuda") for _ in range(2)]
    return s


def _observe(ens, c, obs):
    ix, iy, yu, yv, yr = obs
    if c["rho"]:
        ens.observe_rho(ix, iy, yu, yv, yr, SIGMA, SIGMA, SIGMA_RHO)
    else:
        ens.observe(ix, iy, yu, yv, SIGMA, SIGMA)


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "batch":
        for m in state["members"]:
            m["ens"].set_equilibrium(None, m["x"]["u"], m["x"]["v"])
        state["batch"].cycle(c["steps"], [m["x"]["obs"][:4] + (SIGMA, SIGMA) for m in state["members"]],
                             [m["case"]["d_cut"] for m in state["members"]], [BETA] * len(state["members"]))
        return [m["ens"].get_f(m["out"]) for m in state["members"]]
    ens, x = state["ens"], state["x"]
    if kind == "adjoint":
        J = adjoint.window_misfit(state["f0"], state["cs"], ens, state["win"])
        g, gcs = torch.autograd.grad(J.sum(), (state["f0"], state["cs"]))
        return {"J": J.detach(), "grad_f0": g, "grad_cs": gcs}
    if kind == "diagnostics":
        ens.moments(*state["moments"])
        ens.mean_velocity(*state["mean"])
        ens.energy_spectrum(state["E"])
        return {"rho": state["moments"][0], "u": state["moments"][1], "v": state["moments"][2],
                "um": state["mean"][0], "vm": state["mean"][1], "E": state["E"]}
    if kind == "analysis":
        ens.set_f(x["f"])
    else:
        ens.set_equilibrium(None, x["u"], x["v"])
    if c["steps"]:
        ens.forecast(c["steps"])
        ens.mean_velocity(*state["mean"])
    if kind != "forecast":
        _observe(ens, c, x["obs"])
        ens.analyze(c["d_cut"], BETA)
    out = {"f": ens.get_f(state["out"])}
    if c["steps"]:
        out.update(um=state["mean"][0], vm=state["mean"][1])
    return out


# ---- the same in binary64 torch ---------------------------------------------------

def _moments(f):
    rho = f.sum(0)
    ux = (f[1] - f[2] + f[5] - f[6] + f[7] - f[8]) / rho
    uy = (f[3] - f[4] + f[5] - f[6] - f[7] + f[8]) / rho
    return rho, ux, uy


def _step(f, force, cs):
    """One collide-and-push step; f [9][ny][nx][k]. The non-equilibrium flux
    is sum c c f - rho / 3 I - rho u u (the equilibrium's second moment)."""
    f0, f1, f2, f3, f4, f5, f6, f7, f8 = f.unbind(0)
    s56, s78, d56, d78 = f5 + f6, f7 + f8, f5 - f6, f7 - f8
    sx, sy, diag = f1 + f2, f3 + f4, s56 + s78
    rho = f0 + sx + sy + diag
    jx, jy = f1 - f2 + d56 + d78, f3 - f4 + d56 - d78
    ux, uy = jx / rho, jy / rho
    third = rho / 3.0
    pxx = sx + diag - third - jx * ux
    pyy = sy + diag - third - jy * uy
    pxy = s56 - s78 - jx * uy
    q2 = 2.0 * (pxx * pxx + 2.0 * pxy * pxy + pyy * pyy)
    pos = q2 > 0
    q = torch.where(pos, torch.sqrt(torch.where(pos, q2, 1.0)), 0.0)
    om = 2.0 / (TAU0 + torch.sqrt(TAU0 * TAU0 + 18.0 * cs * cs * q / rho))
    gx, gy = 3.0 * rho * (force[0][:, :, None] - MU * ux), 3.0 * rho * (force[1][:, :, None] - MU * uy)
    base = rho * (1.0 - 1.5 * (ux * ux + uy * uy))
    keep = 1.0 - om
    out = [keep * f0 + om * (W[0] * base)]
    for i, (g, cu, force_a) in enumerate(((f1, ux, gx), (f3, uy, gy), (f5, ux + uy, gx + gy), (f7, ux - uy, gx - gy))):
        w = W[2 * i + 1]
        even = base + 4.5 * rho * cu * cu
        odd = 3.0 * rho * cu
        h = f[2 * i + 2]
        out.append(torch.roll(keep * g + w * (om * (even + odd) + force_a),
                              shifts=(CY[2 * i + 1], CX[2 * i + 1]), dims=(0, 1)))
        out.append(torch.roll(keep * h + w * (om * (even - odd) - force_a),
                              shifts=(CY[2 * i + 2], CX[2 * i + 2]), dims=(0, 1)))
    return torch.stack(out)


def _forecast(f, force, steps):
    for _ in range(steps):
        f = _step(f, force, CS)
    return f


def _weights(c, cells, ix, iy):
    """Gaspari-Cohn weight [cell][point] of the periodic distance."""
    dx = (cells % c["nx"])[:, None] - ix[None, :]
    dy = (cells // c["nx"])[:, None] - iy[None, :]
    dx = torch.minimum(dx % c["nx"], (-dx) % c["nx"]).double()
    dy = torch.minimum(dy % c["ny"], (-dy) % c["ny"]).double()
    d = torch.sqrt(dx * dx + dy * dy) / c["d_cut"]
    near = -0.25 * d ** 5 + 0.5 * d ** 4 + 0.625 * d ** 3 - (5.0 / 3.0) * d * d + 1.0
    e = d.clamp(min=1.0)
    far = e ** 5 / 12.0 - 0.5 * e ** 4 + 0.625 * e ** 3 + (5.0 / 3.0) * e * e - 5.0 * e + 4.0 - (2.0 / 3.0) / e
    w = torch.where(d <= 1.0, near, far)
    return torch.where((d < 2.0) & (w > 0), w, torch.zeros_like(w))


def _inverse_root(C):
    """C^-1/2 of a stack of symmetric positive definite matrices: coupled
    Newton-Schulz iteration on C over a bound of its norm."""
    eye = torch.eye(C.shape[1], dtype=C.dtype, device=C.device)
    s = C.abs().sum(dim=2).amax(dim=1)[:, None, None]
    y, z = C / s, eye.expand_as(C)
    for _ in range(60):
        t = z @ y
        off = float((t - eye).abs().amax())
        t = 1.5 * eye - 0.5 * t
        y, z = y @ t, t @ z
        if off < 1e-9:  # quadratic: the step just made leaves only rounding
            break
    return (z + z.mT) / 2.0 / torch.sqrt(s)


def _analysis(c, f, obs):
    """LETKF analysis of f [9][ny][nx][k] in the ensemble-space form."""
    ix, iy, yu, yv, yr = (torch.as_tensor(np.asarray(o), device="cuda") for o in obs)
    ix, iy, k = ix.long(), iy.long(), c["k"]
    rho, u, v = _moments(f[:, iy, ix, :])
    obs_space = [(u, yu, SIGMA), (v, yv, SIGMA)] + ([(rho, yr, SIGMA_RHO)] if c["rho"] else [])
    outer = torch.zeros((len(ix), k, k), dtype=torch.float64, device="cuda")
    rhs = torch.zeros((len(ix), k), dtype=torch.float64, device="cuda")
    for y, yo, sigma in obs_space:
        dy = y - y.mean(dim=1, keepdim=True)
        outer += dy[:, :, None] * dy[:, None, :] / sigma ** 2
        rhs += dy * (yo - y.mean(dim=1))[:, None] / sigma ** 2
    flat = f.reshape(9, -1, k)
    out = torch.empty_like(flat)
    eye = torch.eye(k, dtype=torch.float64, device="cuda") * ((k - 1) / BETA)
    ncell = flat.shape[1]
    chunk = max(1, min(ncell, 2 ** 26 // (k * k), 2 ** 26 // len(ix)))
    for a in range(0, ncell, chunk):
        cells = torch.arange(a, min(ncell, a + chunk), device="cuda")
        w = _weights(c, cells, ix, iy)
        C = (w @ outer.reshape(len(ix), k * k)).reshape(-1, k, k) + eye
        root = _inverse_root(C)
        wbar = root @ (root @ (w @ rhs)[:, :, None])
        T = wbar + math.sqrt(k - 1.0) * root
        x = flat[:, a:a + chunk].permute(1, 0, 2)
        xm = x.mean(dim=2, keepdim=True)
        out[:, a:a + chunk] = (xm + (x - xm) @ T).permute(1, 0, 2)
    return out.reshape(f.shape)


def _spectrum(u, v):
    ny, nx, k = u.shape
    e = torch.zeros((ny, nx), dtype=torch.float64, device="cuda")
    for w in (u, v):
        e += (torch.fft.fft2(w.permute(2, 0, 1)) / (nx * ny)).abs().square().sum(dim=0) / 2.0 / k
    kx = torch.fft.fftfreq(nx, 1.0 / nx, dtype=torch.float64, device="cuda")[None, :]
    ky = torch.fft.fftfreq(ny, 1.0 / ny, dtype=torch.float64, device="cuda")[:, None]
    shell = torch.floor(torch.sqrt(kx * kx + ky * ky) + 0.5).long().expand(ny, nx)
    return torch.zeros(binding.spectrum_shells(nx, ny), dtype=torch.float64,
                       device="cuda").index_add_(0, shell.reshape(-1), e.reshape(-1))


def _misfit(c, f, cs, force, obs):
    ix, iy, yu, yv, _ = (torch.as_tensor(np.asarray(o), device="cuda") for o in obs)
    ix, iy = ix.long(), iy.long()
    J = torch.zeros(f.shape[3], dtype=torch.float64, device="cuda")

    def one(g, s):
        return _step(g, force, s)

    for t in range(1, c["steps"] + 1):
        f = torch.utils.checkpoint.checkpoint(one, f, cs, use_reentrant=False)
        if t % c["every"] == 0:
            _, u, v = _moments(f[:, iy, ix, :])
            r = t // c["every"] - 1
            J = J + 0.5 * (((u - yu[r][:, None]) / SIGMA) ** 2 + ((v - yv[r][:, None]) / SIGMA) ** 2).sum(0)
    return J


def _too_long(c):
    """Whether the binary64 torch result would take longer than some seconds."""
    cells = c["nx"] * c["ny"]
    if c["kind"] in ("cycle", "analysis"):
        return cells * c["k"] ** 3 > 8e10
    return False


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "batch":
        return [None if _too_long(e) else _exact_one(e, seed, i)["f"] for i, e in enumerate(_experiments(c))]
    return None if _too_long(c) else _exact_one(c, seed, 0)


def _exact_one(c, seed, which):
    x = _inputs(c, seed, which)
    force = torch.as_tensor(x["force"], device="cuda")
    if c["kind"] == "adjoint":
        grads, js, gcs = [], [], 0.0
        for a in range(0, c["k"], 64):
            f0 = x["f"][..., a:a + 64].clone().requires_grad_(True)
            cs = torch.tensor(CS, dtype=torch.float64, device="cuda", requires_grad=True)
            J = _misfit(c, f0, cs, force, x["obs"])
            g, gc = torch.autograd.grad(J.sum(), (f0, cs))
            grads.append(g)
            js.append(J.detach())
            gcs = gcs + gc.cpu()
        return {"J": torch.cat(js), "grad_f0": torch.cat(grads, dim=3), "grad_cs": gcs}
    if c["kind"] == "diagnostics":
        rho, u, v = torch.ones_like(x["u"]), x["u"], x["v"]
        return {"rho": rho, "u": u, "v": v, "um": u.mean(2), "vm": v.mean(2), "E": _spectrum(u, v)}
    f = x["f"] if c["kind"] == "analysis" else _equilibrium(1.0, x["u"], x["v"])
    f = _forecast(f, force, c["steps"])
    out = {}
    if c["steps"]:
        _, u, v = _moments(f)
        out = {"um": u.mean(2), "vm": v.mean(2)}
    if c["kind"] != "forecast":
        f = _analysis(c, f, x["obs"])
    return dict({"f": f}, **out)


# ---- work ----------------------------------------------------------------------

STEP_FLOPS = 150.0  # moments, equilibrium, closure, forcing and relaxation of one member-cell


def _analysis_flops(c):
    """Per grid point with p local scalars and n = min(k, p): 9 n^3 for the
    symmetric eigenproblem and two per multiply-add of the products."""
    ix, iy = inputs.uniform_obs_points(c["nx"], c["ny"], c["nobs_x"], c["nobs_y"])
    yy, xx = np.meshgrid(np.arange(c["ny"]), np.arange(c["nx"]), indexing="ij")
    disc = (np.minimum(xx, c["nx"] - xx) ** 2 + np.minimum(yy, c["ny"] - yy) ** 2 < (2 * c["d_cut"]) ** 2) * 1.0
    pts = np.zeros_like(disc)
    np.add.at(pts, (iy, ix), 1.0)
    cnt = np.rint(np.fft.irfft2(np.fft.rfft2(disc) * np.fft.rfft2(pts), s=disc.shape))
    p, k = (3 if c["rho"] else 2) * cnt, c["k"]
    n = np.minimum(p, k)
    obs = 2 * (p * p + 2 * n * n + 9 * k * p + 2 * 9 * n * n + 9 * k * p)
    ens = 2 * (k * k * p + k * p + 2 * k * k + k ** 3 + 9 * k * k)
    return float(np.sum(9.0 * n ** 3 + np.where(p < k, obs, ens)))


def work(case):
    c = dict(case)
    if c["kind"] == "batch":
        w = [work(e) for e in _experiments(c)]
        return {"bytes": sum(x["bytes"] for x in w), "flops": sum(x["flops"] for x in w)}
    cells = c["nx"] * c["ny"]
    upd = cells * c["k"]
    byts, flops = 16.0 * cells, 0.0
    if c["kind"] == "adjoint":
        byts += 8.0 * 9 * upd * 2
        flops += upd * c["steps"] * 3.0 * STEP_FLOPS
    elif c["kind"] == "diagnostics":
        byts += (9.0 * (8 if c["prec"] == "fp64" else 4) + 3 * 8.0) * upd
        flops += upd * (30.0 + 10.0 * math.log2(cells))
    else:
        byts += 8.0 * 9 * upd + 8.0 * (9 if c["kind"] == "analysis" else 2) * upd + 16.0 * cells
        flops += upd * c["steps"] * STEP_FLOPS
        if c["kind"] != "forecast":
            flops += _analysis_flops(c)
    return {"bytes": byts, "flops": flops}
