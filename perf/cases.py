"""Workloads that the library's speed is measured on.

A case is a dict of plain values; ``prepare`` makes what a user's program holds before the call
(contexts with their medium and state, pinned host arrays), ``run`` is one pass through the public
entry points, ``exact`` the same result from plain torch in 64 bits.  Kinds of case:

  flow      a lattice advanced by ``steps`` steps, then the macroscopic fields (p, ux, uy[, T]); cavities
            with a moving lid, periodic channels, channels between pressure columns, natural
            convection; uniform or per-cell medium; FP32, FP16 and BF16 storage; two population
            buffers or one.  ``monitor`` adds the residual or the Nusselt numbers, which a run to
            steady state reads between its chunks of steps.
  lid       a lattice driven step by step: wall velocities from pinned host memory, one step, a probe
            into pinned host memory, as a coupled or controlled run does.
  ensemble  independent cavities and channels of ragged sizes advanced together.
  gradient  one iteration of a permeability inversion: the loss of a pressure-driven channel after
            ``steps`` steps and its gradient with respect to log K and eps.

Every run starts from a seeded state (smooth waves on top of rest) or a seeded medium.  A flow run may
be repeated: it continues from where the last one ended, as a user's next chunk of steps does.
"""
from __future__ import annotations

import math
import random
from types import SimpleNamespace

import numpy as np
import torch

from paper_1311_7239_gb300 import lbm, workloads

BC = {"periodic": lbm.PERIODIC, "wall": lbm.WALL, "pressure": lbm.PRESSURE, "nee": lbm.NEE}
PREC = {"fp32": lbm.FP32, "fp16": lbm.FP16_DEV, "bf16": lbm.BF16_DEV}
EX = (1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 1, 0, -1, 1, 1, -1, -1)
OPP = (2, 3, 0, 1, 6, 7, 4, 5)
W = (1 / 9,) * 4 + (1 / 36,) * 4
OPP5 = (0, 3, 4, 1, 2)


def _flow(name, nx, ny, steps, prec="fp32", flow="cavity", medium="uniform", streaming="ab", walls="wall", monitor=""):
    return {"name": name, "kind": "flow", "nx": nx, "ny": ny, "steps": steps, "prec": prec, "flow": flow, "medium": medium,
            "streaming": streaming, "walls": walls, "monitor": monitor}


def listed():
    return [
        # the smallest lattice that the accuracy studies step for hundreds of thousands of steps
        _flow("cavity_64", 64, 64, 256),
        # natural convection on a grid of the paper's Table 1, run in chunks between Nusselt read-outs
        _flow("convection_200", 200, 200, 512, flow="convection", monitor="nusselt"),
        # a mid-size porous cavity with a per-cell medium and sides that are no multiple of anything
        _flow("cavity_601x487_medium", 601, 487, 200, medium="cells"),
        # the benchmark's cavity, in each storage precision
        _flow("cavity_4096", 4096, 4096, 100),
        _flow("cavity_4096_fp16", 4096, 4096, 100, prec="fp16"),
        _flow("cavity_1531x1087_bf16", 1531, 1087, 200, prec="bf16"),
        # the natural-convection workload, where the temperature doubles the state
        _flow("convection_2048_fp16", 2048, 2048, 100, prec="fp16", flow="convection"),
        # the forward run of the heterogeneous channel with its convergence check
        _flow("channel_2048x1024_medium", 2048, 1024, 200, flow="pressure", medium="cells", monitor="residual"),
        # the largest lattice, kept in one population buffer for its memory
        _flow("cavity_8192_inplace", 8192, 8192, 32, streaming="inplace"),
        # the smallest calls: one step at a time between host reads and writes
        {"name": "lid_1024_stepwise", "kind": "lid", "nx": 1024, "ny": 1024, "steps": 64, "prec": "fp32"},
        # a batch of independent domains with sides 64..1024
        {"name": "ensemble_48", "kind": "ensemble", "n": 48, "lo": 64, "hi": 1024, "sizes": 42, "steps": 64, "prec": "fp32"},
        # one iteration of the permeability inversion
        {"name": "gradient_2048x1024", "kind": "gradient", "nx": 2048, "ny": 1024, "steps": 100},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["flow"] * 6 + ["lid", "ensemble", "ensemble", "gradient"])
    if kind == "lid":
        return {"kind": kind, "nx": _log_int(rng, 64, 2048), "ny": _log_int(rng, 64, 2048), "steps": rng.randrange(16, 65),
                "prec": rng.choice(["fp32", "fp16"])}
    if kind == "ensemble":
        return {"kind": kind, "n": rng.randrange(8, 49), "lo": 64, "hi": rng.choice([256, 512, 1024]), "sizes": rng.randrange(1 << 20),
                "steps": rng.randrange(16, 65), "prec": rng.choice(["fp32", "fp16", "bf16"])}
    if kind == "gradient":
        return {"kind": kind, "nx": _log_int(rng, 128, 2048), "ny": _log_int(rng, 64, 1024), "steps": rng.randrange(24, 101)}
    nx, ny = _log_int(rng, 48, 4096), _log_int(rng, 48, 4096)
    if rng.random() < 0.4:  # the power-of-two sides of the benchmark's sweep
        nx = ny = 2 ** rng.randrange(6, 13)
    flow = rng.choice(["cavity", "cavity", "periodic", "pressure", "convection"])
    if flow == "convection":
        nx = ny = _log_int(rng, 96, 2048)
    steps = max(16, min(400, int(8e8 / (nx * ny))))
    return {"kind": "flow", "nx": nx, "ny": ny, "steps": rng.randrange(max(16, steps // 2), steps + 1),
            "prec": rng.choice(["fp32", "fp32", "fp16", "bf16"]), "flow": flow,
            "medium": "uniform" if flow == "convection" else rng.choice(["uniform", "cells"]),
            "streaming": rng.choice(["ab", "ab", "ab", "inplace"]),
            "walls": rng.choice(["wall", "wall", "nee"]) if flow in ("cavity", "convection") else "wall",
            "monitor": rng.choice(["", "nusselt" if flow == "convection" else "residual"])}


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
def _waves(gen, ny, nx, modes=5):
    """A smooth field of unit-order amplitude: a few Fourier modes with random phases (float32)."""
    x = torch.arange(nx, dtype=torch.float64, device="cuda") * (2 * math.pi / nx)
    y = torch.arange(ny, dtype=torch.float64, device="cuda") * (2 * math.pi / ny)
    out = torch.zeros(ny, nx, dtype=torch.float32, device="cuda")
    r = torch.rand(modes, 4, generator=gen, dtype=torch.float64).tolist()
    for a, b, c, d in r:
        kx, ky, ph = 1 + int(3 * a), 1 + int(3 * b), 2 * math.pi * c
        u = ((0.5 + d) / modes * torch.cos(ky * y + ph)).float()[:, None]
        out.addcmul_(u, torch.cos(kx * x + 2 * ph).float()[None, :])
    return out


def _random_field(gen, ny, nx, corr):
    """Gaussian random field of correlation length corr, zero mean, unit deviation."""
    noise = torch.randn(ny, nx, generator=gen, device="cuda")
    ky = torch.fft.fftfreq(ny, device="cuda")[:, None]
    kx = torch.fft.rfftfreq(nx, device="cuda")[None, :]
    f = torch.fft.irfft2(torch.fft.rfft2(noise) * torch.exp(-0.5 * (2 * math.pi * corr) ** 2 * (kx * kx + ky * ky)), s=(ny, nx))
    f -= f.mean()
    return f / f.std()


def _medium(seed, ny, nx, da=1e-3):
    """(eps, log K) of a heterogeneous porous medium, float32 [ny, nx]."""
    gen = torch.Generator("cuda").manual_seed(seed)
    corr = min(32.0, max(2.0, min(nx, ny) / 8))
    logk = math.log(da * ny * ny) + _random_field(gen, ny, nx, corr)
    eps = (0.3 + 0.1 * _random_field(gen, ny, nx, corr)).clamp_(0.1, 0.9)
    return eps, logk


def _equilibrium(phip, ux, uy, phi, i):
    eu = EX[i] * ux + EY[i] * uy
    return W[i] * (3.0 * phip + 3.0 * eu + (4.5 * eu * eu - 1.5 * (ux * ux + uy * uy)) / phi)


def _problem(case, seed):
    """Everything that defines a flow case: parameters as plain numbers, fields as float32 tensors."""
    nx, ny = case["nx"], case["ny"]
    q = SimpleNamespace(nx=nx, ny=ny, steps=case["steps"], prec=case["prec"], inplace=case.get("streaming") == "inplace", bc_x="wall",
                        bc_y="wall", nu=0.1, phi=0.4, K=1e-3 * ny * ny, ax=0.0, ay=0.0, lid=(0.0, 0.0), p_in=1.0, p_out=1.0, thermal=None,
                        eps=None, Kf=None, scale=10)
    flow, U = case.get("flow", "cavity"), 0.02
    if case.get("medium") == "cells":
        q.eps, logk = _medium(seed + 1, ny, nx)
        if flow == "pressure":  # the prescribed pressure meets a uniform porosity
            for cols in (slice(0, 4), slice(nx - 4, nx)):
                q.eps[:, cols] = q.eps.mean()
                logk[:, cols] = logk.mean()
        q.Kf = torch.exp(logk)
        q.phi, q.K = float(q.eps.double().mean()), float(torch.exp(logk.double().mean()))
        U = 0.01
    if flow == "cavity":
        q.bc_x = q.bc_y = case.get("walls", "wall")
        q.nu = max(0.1 * min(nx, ny) / 100, 0.02)
        q.lid = (0.02 if q.eps is not None else 0.1, 0.0)
    elif flow == "periodic":
        q.bc_x = "periodic"
        q.ax = 0.01 * q.nu / q.K
    elif flow == "pressure":
        q.bc_x = "pressure"
        dp = min(0.005 * q.nu * (nx - 1) / q.K, 0.04)
        q.p_in, q.p_out = 1.0 + dp / 2, 1.0 - dp / 2
    else:
        c = workloads.natural_convection(lbm, L=nx, Ra=1e6 if nx <= 512 else 1e5, phi=0.6, Da=1e-4 if nx <= 512 else 1e-2)
        q.bc_x = q.bc_y = case.get("walls", "wall")
        q.nu, q.phi, q.K, q.scale = c.nu, c.phi, c.K, c.dev_scale_log2
        q.thermal = SimpleNamespace(zeta=1.0 / c.tau_T, tau=c.tau_T, g_beta=c.g_beta, T0=11.0, walls=(21.0, 1.0, None, None))
    gen = torch.Generator().manual_seed(seed)
    ux, uy, phip = U * _waves(gen, ny, nx), U * _waves(gen, ny, nx), q.phi * (1.0 + 0.01 * _waves(gen, ny, nx))
    phi = q.phi if q.eps is None else q.eps
    q.f0 = torch.empty(8, ny, nx, device="cuda")
    for i in range(8):
        q.f0[i] = _equilibrium(phip, ux, uy, phi, i)
    q.g0 = (0.2 * (11.0 + 4.0 * _waves(gen, ny, nx))).expand(5, ny, nx).contiguous() if q.thermal else None
    return q


def _lattice(q):
    t = q.thermal
    kw = dict(thermal=1, tau_T=t.tau, g_beta=t.g_beta, T0=t.T0, T_wall=list(t.walls)) if t else {}
    lat = lbm.Lattice(nx=q.nx, ny=q.ny, bc_x=BC[q.bc_x], bc_y=BC[q.bc_y], precision=PREC[q.prec], nu=q.nu, phi=q.phi, K=q.K, ax=q.ax,
                      ay=q.ay, u_wall=[(0, 0), (0, 0), (0, 0), q.lid], p_in=q.p_in, p_out=q.p_out, p_rest=q.phi, dev_scale_log2=q.scale,
                      streaming=lbm.STREAM_INPLACE if q.inplace else lbm.STREAM_AB, **kw)
    if q.eps is not None:
        lat.set_medium(q.eps, q.Kf)
    lat.set_populations(q.f0, q.g0)
    return lat


def _lid_problem(case, seed):
    q = _problem({**case, "flow": "cavity"}, seed)
    w = np.zeros((q.steps, 4, 2), np.float32)  # the lid's velocity, step by step
    w[:, 3, 0] = 0.05 + 0.05 * np.sin(0.2 * np.arange(q.steps) + seed % 7)
    q.lid = (float(w[0, 3, 0]), 0.0)
    return q, w


def _domains(case, seed):
    """The lattices of an ensemble: sizes, kinds and Reynolds numbers from the case, media from the seed."""
    r, out = random.Random(case["sizes"]), []
    for d in range(case["n"]):
        nx, ny, cavity, Re = r.randint(case["lo"], case["hi"]), r.randint(case["lo"], case["hi"]), r.random() < 0.5, r.uniform(10, 400)
        out.append((nx, ny, cavity, Re, (seed * 1009 + d) % (1 << 40)))
    return out


def _domain(nx, ny, cavity, Re, seed):
    eps, logk = _medium(seed, ny, nx)
    U = 0.02
    phi, K, nu = float(eps.double().mean()), float(torch.exp(logk.double().mean())), max(U * ny / Re, 0.02)
    x = min(math.sqrt(phi / K) * ny / 2, 300.0)
    return SimpleNamespace(nx=nx, ny=ny, bc_x="wall" if cavity else "periodic", bc_y="wall", nu=nu, phi=phi, K=K, eps=eps,
                           Kf=torch.exp(logk), ax=0.0 if cavity else U * nu / (K * (1.0 - 1.0 / math.cosh(x))), ay=0.0,
                           lid=(U, 0.0) if cavity else (0.0, 0.0), p_in=1.0, p_out=1.0, thermal=None)


def _inversion(case, seed):
    """The pressure-driven channel of the inversion: (parameters, eps, log K)."""
    nx, ny = case["nx"], case["ny"]
    eps, logk = _medium(seed + 1, ny, nx)
    for cols in (slice(0, 4), slice(nx - 4, nx)):
        eps[:, cols] = eps.mean()
        logk[:, cols] = logk.mean()
    phi, K = float(eps.double().mean()), float(torch.exp(logk.double().mean()))
    dp = min(0.01 * 0.1 * (nx - 1) / K, 0.04)
    q = SimpleNamespace(nx=nx, ny=ny, steps=case["steps"], bc_x="pressure", bc_y="wall", nu=0.1, phi=phi, K=K, ax=0.0, ay=0.0,
                        lid=(0.0, 0.0), p_in=1.0 + dp / 2, p_out=1.0 - dp / 2, thermal=None)
    return q, eps, logk


def prepare(case, seed):
    if case["kind"] == "gradient":
        q, eps, logk = _inversion(case, seed)
        cfg = lbm.default_config(nx=q.nx, ny=q.ny, nu=q.nu, phi=q.phi, K=q.K, bc_x=lbm.PRESSURE, bc_y=lbm.WALL, p_in=q.p_in,
                                 p_out=q.p_out, p_rest=q.phi)
        return {"kind": "gradient", "cfg": cfg, "steps": q.steps, "p0": q.phi, "eps": eps.requires_grad_(), "logk": logk.requires_grad_()}
    if case["kind"] == "ensemble":
        qs = [_domain(*d) for d in _domains(case, seed)]
        b = lbm.Batch([lbm.default_config(nx=q.nx, ny=q.ny, nu=q.nu, phi=q.phi, K=q.K, precision=PREC[case["prec"]], p_rest=q.phi, ax=q.ax,
                                          bc_x=BC[q.bc_x], bc_y=BC[q.bc_y], u_wall=[(0, 0), (0, 0), (0, 0), q.lid]) for q in qs])
        for d, q in enumerate(qs):
            b.set_medium(d, q.eps, q.Kf)
            b.init_equilibrium(d, q.phi, 0.0, 0.0, phi_p_uniform=True)
        return {"kind": "ensemble", "batch": b, "steps": case["steps"]}
    if case["kind"] == "lid":
        q, w = _lid_problem(case, seed)
        return {"kind": "lid", "lat": _lattice(q), "walls": torch.from_numpy(w).pin_memory(), "probe": torch.zeros(q.steps, 4).pin_memory(),
                "at": (q.nx // 2, q.ny // 2), "steps": q.steps}
    return {"kind": "flow", "lat": _lattice(_problem(case, seed)), "steps": case["steps"], "monitor": case["monitor"]}


def run(state):
    if state["kind"] == "gradient":
        eps, logk = state["eps"], state["logk"]
        eps.grad = logk.grad = None
        loss = lbm.PorousFlowLoss.apply(logk, eps, state["cfg"], state["steps"], "flux", None, state["p0"], True)
        loss.backward()
        return {"loss": loss.detach().float(), "grad_logk": logk.grad, "grad_eps": eps.grad}
    if state["kind"] == "ensemble":
        b = state["batch"]
        b.step(state["steps"])
        fields = [b.macros(d) for d in range(len(b))]
        return {"p": torch.cat([f[0].reshape(-1) for f in fields]), "u": torch.cat([c.reshape(-1) for f in fields for c in f[1:]])}
    lat = state["lat"]
    u = torch.empty(2, lat.ny, lat.nx, device=lat.device)
    if state["kind"] == "lid":
        (x, y), walls, probe = state["at"], state["walls"], state["probe"]
        for k in range(state["steps"]):
            lat.set_walls(walls[k])
            lat.step(1)
            lat.probe_async(x, y, probe[k])
        p = lat.macros(ux=u[0], uy=u[1])[0]
        lat.sync()  # the probes are read on the host
        return {"p": p, "u": u, "probe": probe.clone()}
    lat.step(state["steps"])
    out = {}
    if state["monitor"] == "residual":
        out["residual"] = np.float32(lat.residual())
    elif state["monitor"] == "nusselt":
        out["nusselt"] = np.float32([lat.nusselt(lbm.LEFT), lat.nusselt(lbm.RIGHT)])
    fields = lat.macros(ux=u[0], uy=u[1])
    out.update(p=fields[0], u=u)
    if lat.thermal:
        out["T"] = fields[3]
    return out


def work(case):
    """Per pass: the stored populations and the medium read once, the populations and the outputs written
    once; 150 operations per cell and step for the flow, 45 more with the temperature, 420 for a
    reverse step."""
    if case["kind"] == "ensemble":
        cells = sum(d[0] * d[1] for d in _domains(case, 0))
    else:
        cells = case["nx"] * case["ny"]
    elem, heat = 4 if case.get("prec", "fp32") == "fp32" else 2, case.get("flow") == "convection"
    if case["kind"] == "gradient":
        return {"bytes": cells * 16.0, "flops": cells * case["steps"] * 570.0}
    medium = 8 if case["kind"] == "ensemble" or case.get("medium") == "cells" else 0
    return {"bytes": cells * (2.0 * (13 if heat else 8) * elem + medium + (16 if heat else 12)),
            "flops": cells * case["steps"] * (195.0 if heat else 150.0)}


# ---------------------------------------------------------------------------------------------
# the same results in 64 bits, from plain torch
# ---------------------------------------------------------------------------------------------
def _velocity(f, q, phi, K, ay):
    """(ux, uy, phi p, |u|, linear drag, nonlinear drag) of pre-collision populations."""
    vx = f[0] - f[2] + f[4] - f[5] - f[6] + f[7] + 0.5 * phi * q.ax
    vy = f[1] - f[3] + f[4] + f[5] - f[6] - f[7] + 0.5 * phi * ay
    lin, non = phi * q.nu / K, 1.75 / torch.sqrt(150.0 * phi * K)
    l0, sq = 0.5 + 0.25 * lin, vx * vx + vy * vy
    v = torch.where(sq > 0, torch.sqrt(torch.where(sq > 0, sq, 1.0)), 0.0)
    d = l0 + torch.sqrt(l0 * l0 + 0.5 * non * v)
    ux, uy = vx / d, vy / d
    return ux, uy, 0.6 * (f.sum(0) - (2.0 / 3.0) * (ux * ux + uy * uy) / phi), v / d, lin, non


def _collide(f, q, phi, K, ay):
    ux, uy, pp, u, lin, non = _velocity(f, q, phi, K, ay)
    Fx, Fy = -(lin + non * u) * ux + phi * q.ax, -(lin + non * u) * uy + phi * ay
    axial, diag = f[:4].sum(0), f[4:].sum(0)
    sv = 1.0 / (0.5 + 3.0 * q.nu)
    k2 = -1.1 * (diag - axial + pp) + 0.45 * 0.8 * (ux * Fx + uy * Fy) / phi
    dx, dy = f[4] - f[5] - f[6] + f[7], f[4] + f[5] - f[6] - f[7]
    k4 = -1.2 * (dx - 2.0 * (f[0] - f[2]) + ux) - 0.4 * Fx
    k6 = -1.2 * (dy - 2.0 * (f[1] - f[3]) + uy) - 0.4 * Fy
    k7 = -sv * (f[0] - f[1] + f[2] - f[3] - (ux * ux - uy * uy) / phi) + (1 - 0.5 * sv) * 2.0 * (ux * Fx - uy * Fy) / phi
    k8 = -sv * (f[4] - f[5] + f[6] - f[7] - ux * uy / phi) + (1 - 0.5 * sv) * (ux * Fy + uy * Fx) / phi
    out = []
    for i in range(8):
        ex, ey = EX[i], EY[i]
        if i < 4:
            k = -k2 / 8 + ex * (Fx / 6 - k4 / 6) + ey * (Fy / 6 - k6 / 6) + (ex * ex - ey * ey) * k7 / 4
        else:
            k = k2 / 8 + ex * (Fx / 6 + k4 / 12) + ey * (Fy / 6 + k6 / 12) + ex * ey * k8 / 4
        out.append(f[i] + k)
    return torch.stack(out), ux, uy


def _stream(fp, q, walls):
    """Streaming of post-collision populations; links through halfway walls bounce back."""
    out = []
    for i in range(8):
        ex, ey, o = EX[i], EY[i], OPP[i]
        s = torch.roll(fp[i], (ey, ex), (0, 1))
        if q.bc_x == "wall" and ex:
            c, w = (0, 0) if ex > 0 else (q.nx - 1, 1)
            s[:, c] = fp[o][:, c] + 6.0 * W[i] * (ex * walls[w][0] + ey * walls[w][1])
        if q.bc_y == "wall" and ey:
            r, w = (0, 2) if ey > 0 else (q.ny - 1, 3)
            s[r] = fp[o][r] + 6.0 * W[i] * (ex * walls[w][0] + ey * walls[w][1])
        out.append(s)
    return torch.stack(out)


def _stream_heat(gp, q):
    t, out = q.thermal, [gp[0]]
    for i, (ex, ey) in enumerate(((1, 0), (0, 1), (-1, 0), (0, -1)), 1):
        s = torch.roll(gp[i], (ey, ex), (0, 1))
        w = {(1, 0): 0, (-1, 0): 1, (0, 1): 2, (0, -1): 3}[ex, ey]
        if (q.bc_x if ex else q.bc_y) == "wall":
            at = (slice(None), 0 if ex > 0 else q.nx - 1) if ex else (0 if ey > 0 else q.ny - 1, slice(None))
            own = gp[OPP5[i]][at]
            s[at] = own if t.walls[w] is None else -own + 0.4 * t.walls[w]
        out.append(s)
    return torch.stack(out)


def _extrapolate(f, g, q, phi, K, walls):
    """Pressure columns and extrapolated wall nodes of a streamed state."""
    t = q.thermal
    if q.bc_x == "pressure":
        f = f.clone()
        for b, n, p in ((0, 1, q.p_in), (q.nx - 1, q.nx - 2, q.p_out)):
            ux, uy, pp = _velocity(f[:, :, n], q, phi[:, n], K[:, n], q.ay)[:3]
            f[:, :, b] = torch.stack([f[i, :, n] + _equilibrium(phi[:, b] * p, ux, uy, phi[:, b], i)
                                      - _equilibrium(pp, ux, uy, phi[:, n], i) for i in range(8)])
    if q.bc_x != "nee" and q.bc_y != "nee":
        return f, g
    fn, gn = f, g
    f, g = f.clone(), None if g is None else g.clone()
    inner = list(range(q.nx))
    if q.bc_x == "nee":
        inner[0], inner[-1] = 1, q.nx - 2
    ally, allx = torch.arange(q.ny, device=f.device), torch.arange(q.nx, device=f.device)
    inx = torch.tensor(inner, device=f.device)
    sides = []
    if q.bc_x == "nee":
        sides += [(ally, allx[:1], ally, allx[1:2], 0), (ally, allx[-1:], ally, allx[-2:-1], 1)]
    if q.bc_y == "nee":  # bottom and top walls own the corners
        sides += [(ally[:1], allx, ally[1:2], inx, 2), (ally[-1:], allx, ally[-2:-1], inx, 3)]
    for yb, xb, yn, xn, w in sides:
        at, nb = (yb[:, None], xb[None, :]), (yn[:, None], xn[None, :])
        pb, pn = phi[at], phi[nb]
        d = torch.stack([fn[i][nb] for i in range(8)])
        ay = q.ay
        if t:
            e = torch.stack([gn[i][nb] for i in range(5)])
            T = e.sum(0)
            ay = q.ay + t.g_beta * (T - t.T0)
        ux, uy, pp = _velocity(d, q, pn, K[nb], ay)[:3]
        wx, wy = (torch.full_like(ux, float(c)) for c in walls[w])
        for i in range(8):
            f[i][at] = d[i] + _equilibrium(pp * pb / pn, wx, wy, pb, i) - _equilibrium(pp, ux, uy, pn, i)
        if t:
            Tb = T if t.walls[w] is None else torch.full_like(T, t.walls[w])
            for i, (ex, ey) in enumerate(((0, 0), (1, 0), (0, 1), (-1, 0), (0, -1))):
                g[i][at] = e[i] + 0.2 * (Tb - T) + 0.5 * ((ex * wx + ey * wy) * Tb - (ex * ux + ey * uy) * T)
    return f, g


def _collide_heat(g, ux, uy, q):
    T, t = g.sum(0), q.thermal
    r1, r2 = -0.5 * t.zeta * (g[1] - g[3] - ux * T), -0.5 * t.zeta * (g[2] - g[4] - uy * T)
    r3, r4 = -0.055 * (g[1:].sum(0) - 4.0 * g[0]), -0.275 * (g[1] - g[2] + g[3] - g[4])
    return torch.stack([g[0] - 4.0 * r3, g[1] + r1 + r3 + r4, g[2] + r2 + r3 - r4, g[3] - r1 + r3 + r4, g[4] - r2 + r3 - r4])


def _advance(f, g, q, phi, K, walls):
    """One step of a pre-collision state: collision, streaming, boundary nodes."""
    ay = q.ay if g is None else q.ay + q.thermal.g_beta * (g.sum(0) - q.thermal.T0)
    f, ux, uy = _collide(f, q, phi, K, ay)
    if g is not None:
        g = _stream_heat(_collide_heat(g, ux, uy, q), q)
    return _extrapolate(_stream(f, q, walls), g, q, phi, K, walls)


def _fields(f, g, q, phi, K):
    ay = q.ay if g is None else q.ay + q.thermal.g_beta * (g.sum(0) - q.thermal.T0)
    ux, uy, pp = _velocity(f, q, phi, K, ay)[:3]
    return [pp / phi, ux, uy] + ([] if g is None else [g.sum(0)])


def _double(q):
    full = torch.ones(q.ny, q.nx, dtype=torch.float64, device="cuda")
    uniform = getattr(q, "eps", None) is None
    return (full * q.phi, full * q.K) if uniform else (q.eps.double(), q.Kf.double())


def _nusselt(T, q):
    """Mean temperature gradients at the isothermal walls times width over temperature difference."""
    out = []
    for s, (Tw, sign) in enumerate(((21.0, -1.0), (1.0, 1.0))):
        a, b, c = (T[:, k if s == 0 else -1 - k] for k in range(3))
        if q.bc_x == "nee":
            out.append(sign * ((-3 * a + 4 * b - c) / 2)[1:-1].mean() * (q.nx - 1) / 20.0)
        else:
            out.append(sign * ((9 * a - b - 8 * Tw) / 3).mean() * q.nx / 20.0)
    return torch.stack(out)


def exact(case, seed):
    if case["kind"] == "gradient":
        return _exact_gradient(case, seed)
    if case["kind"] == "ensemble":
        p, u = [], []
        for d in _domains(case, seed):
            q = _domain(*d)
            phi, K = _double(q)
            zero = torch.zeros_like(phi)
            f = torch.stack([_equilibrium(q.phi + zero, zero, zero, phi, i) for i in range(8)])
            for _ in range(case["steps"]):
                f = _advance(f, None, q, phi, K, ((0, 0), (0, 0), (0, 0), q.lid))[0]
            r = _fields(f, None, q, phi, K)
            p.append(r[0].reshape(-1))
            u += [r[1].reshape(-1), r[2].reshape(-1)]
        return {"p": torch.cat(p), "u": torch.cat(u)}
    if case["kind"] == "lid":
        q, w = _lid_problem(case, seed)
        phi, K = _double(q)
        f, w, probe = q.f0.double(), w.astype(np.float64), []
        for k in range(q.steps):
            post = _collide(f, q, phi, K, 0.0)[0]
            now = _fields(_stream(post, q, w[k]), None, q, phi, K)
            probe.append(torch.stack([c[q.ny // 2, q.nx // 2] for c in now] + [torch.zeros((), device="cuda")]))
            f = _stream(post, q, w[min(k + 1, q.steps - 1)])  # the wall velocity set before the next step
        return {"p": now[0], "u": torch.stack(now[1:]), "probe": torch.stack(probe)}
    q = _problem(case, seed)
    phi, K = _double(q)
    walls = ((0, 0), (0, 0), (0, 0), q.lid)
    f, g = _extrapolate(q.f0.double(), None if q.g0 is None else q.g0.double(), q, phi, K, walls)
    q.f0 = q.g0 = None
    for k in range(q.steps):
        if k == q.steps - 1 and case["monitor"] == "residual":
            before = _fields(f, g, q, phi, K)
        f, g = _advance(f, g, q, phi, K, walls)
    r = _fields(f, g, q, phi, K)
    out = {"p": r[0], "u": torch.stack(r[1:3])}
    if g is not None:
        out["T"] = r[3]
    if case["monitor"] == "residual":
        out["residual"] = torch.sqrt(((r[1] - before[1]) ** 2 + (r[2] - before[2]) ** 2).sum() / (r[1] ** 2 + r[2] ** 2).sum())
    elif case["monitor"] == "nusselt":
        out["nusselt"] = _nusselt(r[3], q)
    return out


def _exact_gradient(case, seed):
    from torch.utils.checkpoint import checkpoint

    q, eps, logk = _inversion(case, seed)
    phi, lk = eps.double().requires_grad_(), logk.double().requires_grad_()
    K, walls = torch.exp(lk), ((0, 0),) * 4
    zero = torch.zeros_like(phi)
    f = torch.stack([_equilibrium(q.phi + zero, zero, zero, phi, i) for i in range(8)])
    f = _extrapolate(f, None, q, phi, K, walls)[0]

    def step(f, phi, K):
        return _advance(f, None, q, phi, K, walls)[0]

    for _ in range(q.steps):
        f = checkpoint(step, f, phi, K, use_reentrant=False)
    loss = _velocity(f, q, phi, K, 0.0)[0][:, -1].sum()
    loss.backward()
    return {"loss": loss.detach(), "grad_logk": lk.grad, "grad_eps": phi.grad}
