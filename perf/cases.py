"""What a user of this framework has it do, as measurable cases over the public entry points.

Every case goes through ``paper_2608_13437_gb300.lbm`` (``Domain``, ``Batch`` and, for the
per-domain outputs of a batch on the device, the C ABI's ``lbm_batch_moments``) or
``paper_2608_13437_gb300.spectral``. The problems are those of ``inputs.py``: the Sod tube
with held ends, the supersonic Taylor-Green vortex (TGV) and smooth random states; initial
fields are made from the seed on the GPU (or on the host where the call takes host arrays).

``exact`` restates the scheme in FP64 with plain torch operations (D3Q7 per field, linear
equilibrium, BGK with the blended rate, explicit source, streaming by rolls).
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2608_13437_gb300 import inputs, lbm, spectral

L2_BYTES = 129e6       # on-chip L2 of the GB300
FLOPS_PER_CELL = 950   # FP32 operations of one cell update (moments, closure, flux, collision)
MOST_UPDATES = 6e8     # cell updates of a drawn case (march512_f32: 8.1e8)
ES = {"f32": 4, "f16": 2, "bf16": 2}


# ------------------------------------------------------------------------------- the cases
def listed():
    def c(name, kind, nx, ny, nz, store, steps, streaming=0, sr=0, **more):
        return dict(name=name, kind=kind, nx=nx, ny=ny, nz=nz, store=store, steps=steps,
                    streaming=streaming, sr=sr, **more)

    return [
        # Sec. 3.1's shock tube at the size the tests run, to its end time 0.2: 16 thousand
        # cells and 1282 steps, the smallest grid in earnest use; launches and latency count.
        c("sod1024_f32", "sod", 1024, 4, 4, "f32", 1282),
        # The parity configuration: 32^3, 100 steps from caller fields, all 14 moments read.
        c("tgv32_f32", "run", 32, 32, 32, "f32", 100),
        # A dissipation time series at the coarsest size the paper lists: a diagnostic sample
        # every 100 steps (tgv_series' default), 16-bit storage.
        c("series64_f16", "series", 64, 64, 64, "f16", 100, samples=3),
        # Sides that are no multiples of the 32-cell tile, smooth flow, 16-bit storage.
        c("ragged150x100x60_bf16", "run", 150, 100, 60, "bf16", 50),
        # A job as README shows it, on host arrays: fields in, steps, diag(), primitives().
        c("job96_f32", "job", 96, 96, 96, "f32", 50),
        # A sampled run at 128^3 (the drift study's size), esoteric twist.
        c("series128_f32", "series", 128, 128, 128, "f32", 20, streaming=1, samples=3),
        # An ordinary production size with stochastic rounding, esoteric twist, mid-run.
        c("march256_bf16_sr", "march", 256, 256, 256, "bf16", 20, streaming=1, sr=1),
        # The benchmark's domain, mid-run: 52.6 GB of state.
        c("march512_f32", "march", 512, 512, 512, "f32", 6, streaming=1),
        # The benchmark's 64 seeded domains of 32^3 to 128^3 in one batch, 16-bit storage.
        dict(name="batch64_f16", kind="batch", store="f16", steps=8, streaming=0, sr=0,
             sizes=",".join(str(d["n"]) for d in inputs.batch_domains(64, 0))),
        # Looking at a state: lbm_diag as a pass of its own, and all moments on the device.
        c("snapshot256_f16", "snapshot", 256, 256, 256, "f16", 4),
        # Restart: canonical populations to the host and into another handle, bit for bit.
        c("restart64_f32", "restart", 64, 64, 64, "f32", 5),
        # Spectral sample of a run (Eq. 7 and E(k) as the paper evaluates them).
        c("spectral128_f32", "spectral", 128, 128, 128, "f32", 4, streaming=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same kinds: sizes over the logarithm of each kind's range, odd and
    ragged ones among them, any storage type, rounding and streaming map."""
    kind = rng.choice(["sod", "run", "run", "series", "job", "march", "batch", "snapshot",
                       "restart", "spectral"])
    store = rng.choice(["f32", "f16", "bf16"])
    c = dict(kind=kind, store=store, streaming=rng.randrange(2),
             sr=rng.randrange(2) if store != "f32" else 0)
    if kind == "sod":
        n = _log(rng, 64, 4096)
        c.update(nx=n, ny=rng.choice([1, 2, 4, 6]), nz=rng.choice([1, 3, 4]),
                 steps=min(_log(rng, 60, 1500), 5 * n // 4))  # no wave has reached an end
        return c
    if kind == "batch":
        n = _log(rng, 4, 64)
        sides = [rng.choice((20, 32, 33, 48, 64, 96, 128)) for _ in range(n)]
        c.update(sizes=",".join(map(str, sides)),
                 steps=min(rng.randrange(4, 13), max(2, int(MOST_UPDATES / sum(v ** 3 for v in sides)))))
        return c
    lo, hi = {"run": (16, 224), "series": (24, 160), "job": (24, 112), "march": (160, 352),
              "snapshot": (32, 320), "restart": (16, 72), "spectral": (32, 144)}[kind]
    n = _log(rng, lo, hi)
    c.update(nx=n, ny=n, nz=n, steps={"run": _log(rng, 10, 100), "series": _log(rng, 10, 100),
                                      "job": _log(rng, 10, 60), "march": rng.randrange(4, 17)}.get(kind, 3))
    if kind in ("run", "job", "snapshot", "restart", "march") and rng.random() < 0.6:
        # a box: two more sides, each drawn, about the same number of cells at most
        c.update(ny=max(8, _log(rng, lo / 2, n)), nz=max(8, _log(rng, lo / 2, n)))
    if kind == "series":
        c["samples"] = rng.randrange(1, 4)
    most = MOST_UPDATES / (c["nx"] * c["ny"] * c["nz"] * c.get("samples", 1))
    c["steps"] = max(1, min(c["steps"], int(most)))
    return c


# ------------------------------------------------------------------------------- inputs
def _generator(seed, device="cuda"):
    return torch.Generator(device=device).manual_seed(int(seed))


def _cube(case):
    return case["nx"] == case["ny"] == case["nz"]


def _params(case):
    if case["kind"] == "sod":
        p = inputs.sod_params(case["nx"], ny=case["ny"], nz=case["nz"])
    elif _cube(case):
        p = inputs.tgv_params(case["nx"])
    else:  # smooth flow in a box, as the ragged-size tests set it
        p = inputs.tgv_params(32)
        p.update(nx=case["nx"], ny=case["ny"], nz=case["nz"], dx=2 * math.pi / case["nx"],
                 sutherland=0, f_mu=0.3, J_min=1e-3, tau_R=0.05, tau_q=0.05)
    return dict(p, streaming=case["streaming"], stochastic_round=case["sr"])


def _fields(case, seed):
    """rho, u, p (5, nz, ny, nx) float32 on the GPU: in a cube the supersonic TGV (Sec. 3.2),
    shifted and carried by a wind that the seed draws, with a compressive wave per axis (a
    state of a run is not free of divergence); in a box a smooth state of low modes."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    r = np.random.default_rng(int(seed))

    def axis(n, d):
        shape = [1, 1, 1]
        shape[d] = n
        return (torch.arange(n, device="cuda", dtype=torch.float32) * (2 * math.pi / n)).view(shape)

    ph = r.uniform(0, 2 * math.pi, 3)
    x, y, z = axis(nx, 2) + ph[0], axis(ny, 1) + ph[1], axis(nz, 0) + ph[2]
    wind = r.uniform(0.05, 0.15, 3)
    out = torch.empty((5, nz, ny, nx), dtype=torch.float32, device="cuda")
    if _cube(case):
        M0 = 1.25
        p0 = 1.0 / (inputs.GAMMA * M0 * M0)
        out[4] = p0 + (torch.cos(2 * x) + torch.cos(2 * y)) * (torch.cos(2 * z) + 2.0) / 16.0
        out[0] = out[4] / p0
        out[1] = wind[0] + torch.sin(x) * torch.cos(y) * torch.cos(z) + 0.2 * torch.cos(x)
        out[2] = wind[1] - torch.cos(x) * torch.sin(y) * torch.cos(z) + 0.2 * torch.cos(y)
        out[3] = wind[2] + 0.2 * torch.cos(z)
        return out
    for j, base in enumerate((1.0, wind[0], wind[1], wind[2], 1.0)):
        out[j] = base
        for _ in range(3):
            k = r.integers(0, 3, 3)
            out[j] += 0.033 * r.standard_normal() * torch.sin(
                float(k[0]) * x + float(k[1]) * y + float(k[2]) * z + r.uniform(0, 6.28))
    return out


def _sod_states(seed):
    """Left and right (rho, u, p): Sec. 3.1's, each value within 2 %."""
    r = np.random.default_rng(int(seed))
    j = 1 + 0.02 * r.uniform(-1, 1, 4)
    return (1.0 * j[0], 0.0, 1.0 * j[1]), (0.125 * j[2], 0.0, 0.1 * j[3])


def _batch_problem(case, seed):
    """Per domain: side, M0, Re, U0, rho0 (M0 below the near-vacuum limit of the TGV)."""
    r = np.random.default_rng(int(seed))
    return [dict(n=int(n), M0=float(r.uniform(0.3, 1.3)), Re=float(r.uniform(100.0, 1600.0)),
                 U0=float(r.uniform(0.9, 1.1)), rho0=float(r.uniform(0.9, 1.1)))
            for n in case["sizes"].split(",")]


def _batch_params(case, d):
    p = inputs.tgv_params(d["n"], M0=d["M0"], Re=d["Re"], U0=d["U0"], rho0=d["rho0"])
    return dict(p, streaming=case["streaming"], stochastic_round=case["sr"])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        ds = _batch_problem(case, seed)
        b = lbm.Batch([_batch_params(case, d) for d in ds], store=case["store"])
        b.init_tgv([d["U0"] for d in ds], [d["M0"] for d in ds], [d["rho0"] for d in ds])
        out = [torch.empty((6,) + (d["n"],) * 3, device="cuda") for d in ds]
        return dict(case=case, batch=b, out=out)
    dom = lbm.Domain(_params(case), store=case["store"])
    s = dict(case=case, dom=dom)
    if kind == "sod":
        s["left"], s["right"] = _sod_states(seed)
        return s
    fields = _fields(case, seed)
    if kind in ("run", "series") and not _evolves(case):
        s["fields"] = fields
        return s
    if kind == "job":
        s["fields"] = fields.double().cpu().numpy()
        return s
    dom.init_fields_device(fields)
    if kind in ("snapshot", "restart", "spectral"):  # a state some steps into a run
        dom.step(case["steps"])
    if kind == "restart":
        s["other"] = lbm.Domain(_params(case), store=case["store"])
        s["other"].init_fields_device(fields)
    return s


def _evolves(case):
    """Whether a pass continues the run of the one before (larger grids); on smaller ones a
    pass is a whole short run from its initial fields."""
    return case["kind"] == "march" or (case["kind"] == "series" and case["nx"] > 100)


# ------------------------------------------------------------------------------- one pass
def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "batch":
        b = s["batch"]
        b.step(case["steps"])
        for d, out in enumerate(s["out"]):
            lbm.check(lbm.lib().lbm_batch_moments(b._h, d, lbm.MOM_PRIM,
                                                  ctypes.c_void_p(out.data_ptr()), 1, lbm.DT_F32))
        return s["out"]
    dom = s["dom"]
    if kind == "sod":
        dom.init_riemann(0, case["nx"] // 2, s["left"], s["right"])
        dom.step(case["steps"])
        return dom.moments_device(lbm.MOM_PRIM)
    if kind == "run":
        dom.init_fields_device(s["fields"])
        dom.step(case["steps"])
        return dom.moments_device()
    if kind == "series":
        if not _evolves(case):
            dom.init_fields_device(s["fields"])
        samples = [dom.step_diag(case["steps"]) for _ in range(case["samples"])]
        return {"samples": samples, "prim": dom.moments_device(lbm.MOM_PRIM)}
    if kind == "march":
        dom.step(case["steps"])
        return dom.moments_device(lbm.MOM_PRIM)
    if kind == "job":
        rho, ux, uy, uz, p = s["fields"]
        dom.init_fields(rho, ux, uy, uz, p)
        dom.step(case["steps"])
        return {"diag": dom.diag(), "prim": dom.primitives()}
    if kind == "snapshot":
        return {"diag": dom.diag(), "q": dom.moments_device()}
    if kind == "restart":
        pops = dom.populations("native")
        s["other"].set_populations(pops, native=True)
        return {"populations": pops, "q": s["other"].moments_device()}
    # spectral: as tgv_series samples a run
    p = dom.params
    prim = dom.moments_device(lbm.MOM_PRIM, torch.float64)
    eps_s, eps_d = spectral.dissipation(prim, p["mu"], p["T_ref"], p["sutherland"], 1.0)
    k, e = spectral.energy_spectrum(prim[1:4])
    return {"eps_s": eps_s, "eps_d": eps_d, "E": e, "prim": prim}


def work(case):
    """What a pass cannot do without: inputs read and outputs written once, and the state of
    98 populations per cell read and written once per step, unless it fits the L2 (then once
    per pass: nothing forces it off the chip between the steps)."""
    kind, es, steps = case["kind"], ES[case["store"]], case["steps"]
    sides = [[int(n)] * 3 for n in case["sizes"].split(",")] if kind == "batch" else \
        [[case["nx"], case["ny"], case["nz"]]]
    cells = sum(a * b * c for a, b, c in sides)
    state = 98 * es * cells
    if kind in ("snapshot", "restart", "spectral"):
        out = {"snapshot": state + state + 56 * cells, "restart": 4 * state + state + 56 * cells,
               "spectral": state + 48 * cells + 48 * cells}[kind]
        per = {"snapshot": 300, "restart": 100,
               # 3 transforms forward and 4 back of a real field, and the spectrum's sums
               "spectral": 7 * 2.5 * math.log2(max(2, cells)) + 100}[kind]
        return {"bytes": out, "flops": per * cells}
    passes = steps * (case["samples"] if kind == "series" else 1)
    moved = 2 * state * (passes if state > L2_BYTES else 1)
    io = {"sod": 24, "run": 20 + 56, "series": 24, "march": 24, "job": 40 + 48, "batch": 24}[kind] * cells
    if kind == "job":
        moved += state  # the diagnostic pass
    return {"bytes": moved + io, "flops": FLOPS_PER_CELL * cells * passes}


# ------------------------------------------------------------------------------- FP64
class _Fp64:
    """The scheme in FP64 by plain tensor operations: f (14, 7, nz, ny, nx)."""

    AXES = (-1, -2, -3)  # x, y, z

    def __init__(self, p, rho, u, pr):
        self.p = p
        self.dt = p["dt"] if p["dt"] > 0 else p["cfl"] * 0.5 * p["dx"] / p["lambda_ref"]
        unit = self.dt if p["relax_in_dt"] else 1.0
        self.tau_R, self.tau_q = p["tau_R"] * unit, p["tau_q"] * unit
        self.c = p["dx"] / self.dt
        self.steps = 0
        E = pr / (p["gamma"] - 1) + 0.5 * rho * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
        zero = torch.zeros_like(rho)
        Q = [rho, rho * u[0], rho * u[1], rho * u[2], E] + [zero] * 9
        s = self.closure(Q)
        self.f = torch.empty((14, 7) + tuple(rho.shape), dtype=torch.float64, device=rho.device)
        for k in range(14):
            phi = self.flux(k, s)
            self.f[k, 0] = Q[k] / 4
            for a in range(3):
                self.f[k, 1 + 2 * a] = Q[k] / 8 + phi[a] / (2 * self.c)
                self.f[k, 2 + 2 * a] = Q[k] / 8 - phi[a] / (2 * self.c)
        self.ghost = (self.f[:, 1, :, :, 0].clone(), self.f[:, 2, :, :, -1].clone()) if p["bc_x"] else None

    def closure(self, Q):
        p = self.p
        rho, m, E = Q[0], Q[1:4], Q[4]
        u = [v / rho for v in m]
        pr = (p["gamma"] - 1) * (E - 0.5 * (m[0] * u[0] + m[1] * u[1] + m[2] * u[2]))
        T = pr / rho
        ratio = torch.ones_like(T)
        if p["sutherland"]:
            t = T / p["T_ref"]
            ratio = 1.4042 * t * torch.sqrt(t) / (t + 0.4042)
        tau = {(0, 0): Q[5], (1, 1): Q[6], (2, 2): Q[7], (0, 1): Q[8], (0, 2): Q[9], (1, 2): Q[10]}
        return dict(rho=rho, m=m, u=u, E=E, p=pr, T=T, mu=p["mu"] * ratio, tau=tau, q=Q[11:14],
                    visc=p["mu"] / self.tau_R * ratio, heat=p["kappa"] / self.tau_q * ratio)

    PAIRS = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))

    def flux(self, k, s):
        u, m, tau = s["u"], s["m"], s["tau"]

        def t(a, b):
            return tau[(min(a, b), max(a, b))]

        if k == 0:
            return m
        if k <= 3:
            b = k - 1
            return [m[b] * u[a] - t(a, b) + (s["p"] if a == b else 0) for a in range(3)]
        if k == 4:
            return [(s["E"] + s["p"]) * u[a] - sum(t(a, b) * u[b] for b in range(3)) + s["q"][a]
                    for a in range(3)]
        if k <= 10:
            b, c = self.PAIRS[k - 5]
            out = []
            for a in range(3):
                lam = (u[c] if a == b else 0) + (u[b] if a == c else 0) - (2 / 3 * u[a] if b == c else 0)
                out.append(t(b, c) * u[a] - s["visc"] * lam)
            return out
        b = k - 11
        return [s["q"][b] * u[a] + (s["heat"] * s["T"] if a == b else 0) for a in range(3)]

    def moments(self):
        return [self.f[k].sum(0) for k in range(14)]

    def step(self, n=1):
        for _ in range(n):
            self._one()

    def _one(self):
        p, f, c, dt = self.p, self.f, self.c, self.dt
        Q = self.moments()
        s = self.closure(Q)
        rho, u, m = s["rho"], s["u"], s["m"]
        omega = 1 / (0.5 + 4 * p["f_mu"] * s["mu"] / rho * dt / p["dx"] ** 2)
        acc = f[0, 0] - rho / 4
        for a in range(3):
            fneq = f[1 + a, 0] - m[a] / 4
            acc = acc - u[a] / c * (4 * fneq / c - (f[0, 1 + 2 * a] - f[0, 2 + 2 * a]) + m[a] / c)
        theta = 4 * omega / rho * acc
        mach = 2 * torch.clamp(-theta, min=0)
        chi = torch.where(mach > p["J_min"], torch.clamp(p["C_sigma"] * mach, max=1.0),
                          torch.zeros_like(mach))
        om = omega - chi * (omega - p["omega_min"])
        for k in range(14):
            phi = self.flux(k, s)
            src = 0 if k < 5 else -dt / (self.tau_R if k < 11 else self.tau_q)
            f[k, 0] += om * (Q[k] / 4 - f[k, 0]) + src * Q[k] / 4
            for a in range(3):
                for i, sign in ((1 + 2 * a, 1), (2 + 2 * a, -1)):
                    g = f[k, i] + om * (Q[k] / 8 + sign * phi[a] / (2 * c) - f[k, i]) + src * Q[k] / 8
                    f[k, i] = torch.roll(g, sign, self.AXES[a])
        if self.ghost is not None:
            f[:, 1, :, :, 0], f[:, 2, :, :, -1] = self.ghost
        self.steps += 1

    def prim(self):
        s = self.closure(self.moments())
        return torch.stack([s["rho"], *s["u"], s["T"], s["p"]])

    def diag(self):
        p = self.p
        s = self.closure(self.moments())
        rho, u, T = s["rho"], s["u"], s["T"]

        def d(b, a):  # central difference of u_b along a
            return (torch.roll(u[b], -1, self.AXES[a]) - torch.roll(u[b], 1, self.AXES[a])) / (2 * p["dx"])

        w2 = (d(2, 1) - d(1, 2)) ** 2 + (d(0, 2) - d(2, 0)) ** 2 + (d(1, 0) - d(0, 1)) ** 2
        div = d(0, 0) + d(1, 1) + d(2, 2)
        u2 = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        a = torch.sqrt(p["gamma"] * T)
        umax = torch.stack([v.abs() for v in u]).amax(0)
        vals = dict(step=self.steps, time=self.steps * self.dt, sum_rho=rho.sum(), sum_mx=s["m"][0].sum(),
                    sum_my=s["m"][1].sum(), sum_mz=s["m"][2].sum(), sum_E=s["E"].sum(),
                    ek_mean=(0.5 * rho * u2).mean(), eps_s_raw=(s["mu"] * w2).mean(),
                    eps_d_raw=4 / 3 * (s["mu"] * div ** 2).mean(),
                    max_mach=(torch.sqrt(u2) / a).max(), max_cfl=(umax + a).max() * self.dt / p["dx"],
                    min_rho=rho.min(), min_T=T.min(), nonfinite=0)
        return {k: float(v) for k, v in vals.items()}


def exact(case, seed):
    """run()'s outputs for the seed's inputs in FP64; None where the grid is too large for it."""
    kind, steps = case["kind"], case["steps"]

    def numbers(o):  # 8-bit mantissas: the noise of the divergence swamps its mean square
        return dict(o.diag(), status=None, **({"eps_d_raw": None} if case["store"] == "bf16" else {}))

    if kind == "batch":
        out = []
        for d in _batch_problem(case, seed):
            n, h = d["n"], 2 * math.pi / d["n"]
            r = torch.arange(n, device="cuda", dtype=torch.float64) * h
            x, y, z = r.view(1, 1, n), r.view(1, n, 1), r.view(n, 1, 1)
            p0 = d["rho0"] * d["U0"] ** 2 / (inputs.GAMMA * d["M0"] ** 2)
            pr = p0 + d["rho0"] * d["U0"] ** 2 / 16 * (torch.cos(2 * x) + torch.cos(2 * y)) * (torch.cos(2 * z) + 2)
            u = [d["U0"] * torch.sin(x) * torch.cos(y) * torch.cos(z),
                 -d["U0"] * torch.cos(x) * torch.sin(y) * torch.cos(z), torch.zeros_like(pr)]
            o = _Fp64(_batch_params(case, d), pr / p0 * d["rho0"], u, pr)
            o.step(steps)
            out.append(o.prim())
        return out
    p = _params(case)
    if case["nx"] * case["ny"] * case["nz"] > 20e6:
        return None
    if kind == "sod":
        left, right = _sod_states(seed)
        side = (torch.arange(case["nx"], device="cuda") < case["nx"] // 2).expand(case["nz"], case["ny"], -1)
        rho, u, pr = (torch.where(side, torch.tensor(left[j], dtype=torch.float64, device="cuda"),
                                  torch.tensor(right[j], dtype=torch.float64, device="cuda")) for j in range(3))
        o = _Fp64(p, rho, [u, torch.zeros_like(u), torch.zeros_like(u)], pr)
        o.step(steps)
        return o.prim()
    f = _fields(case, seed).double()
    o = _Fp64(p, f[0], f[1:4], f[4])
    del f
    if kind == "series":
        samples = []
        for _ in range(case["samples"]):
            samples.append(numbers(o))
            o.step(steps)
        return {"samples": samples, "prim": o.prim()}
    o.step(steps)
    if kind == "run":
        return torch.stack(o.moments())
    if kind == "march":
        return o.prim()
    if kind == "job":
        return {"diag": numbers(o), "prim": o.prim()}
    if kind == "snapshot":
        return {"diag": numbers(o), "q": torch.stack(o.moments())}
    if kind == "restart":
        return {"populations": None, "q": torch.stack(o.moments())}
    prim = o.prim()
    e = dict(_spectra(prim, p), prim=prim)
    return dict(e, eps_d=None) if case["store"] == "bf16" else e


def _spectra(prim, p):
    """eps_s, eps_d of Eq. 7 and E(k) over unit shells, by FP64 transforms."""
    nz, ny, nx = prim.shape[1:]
    k = [torch.fft.fftfreq(n, d=1.0 / n, device="cuda", dtype=torch.float64) for n in (nx, ny, nz)]
    grid = [k[0].view(1, 1, nx), k[1].view(1, ny, 1), k[2].view(nz, 1, 1)]
    uh = [torch.fft.fftn(prim[1 + b]) for b in range(3)]
    shell = torch.round(torch.sqrt(grid[0] ** 2 + grid[1] ** 2 + grid[2] ** 2)).long().reshape(-1)
    e = sum(0.5 * (v.abs() / v.numel()) ** 2 for v in uh).reshape(-1)
    E = torch.bincount(shell, weights=e)

    def d(b, a):
        ka = torch.where(grid[a].abs() * 2 == prim.shape[3 - a], torch.zeros_like(grid[a]), grid[a])
        return torch.fft.ifftn(1j * ka * uh[b]).real

    T = prim[4] / p["T_ref"]
    mu = p["mu"] * 1.4042 * T ** 1.5 / (T + 0.4042) if p["sutherland"] else p["mu"] + 0 * T
    w2 = (d(2, 1) - d(1, 2)) ** 2 + (d(0, 2) - d(2, 0)) ** 2 + (d(1, 0) - d(0, 1)) ** 2
    div = d(0, 0) + d(1, 1) + d(2, 2)
    return {"eps_s": float((mu * w2).mean()), "eps_d": float(4 / 3 * (mu * div ** 2).mean()), "E": E}
