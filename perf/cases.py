"""Workloads of the JFNK library, timed through its public entry points.

A case is a plain dict; ``prepare`` makes what a user's program holds before
the call (state, inputs, solver handle), ``run`` is one pass and returns all
that the call computes, ``exact`` is the same result in 64 bits by plain torch
(its own discretisation and solver, nothing of this package's numerics).

Kinds of case
    operators     F(u) and the trapezoidal residual R(u^n, u) in float64:
                  what a program calls to monitor or couple a model
    step          one implicit step u^n -> u^{n+1} on device data
    batch         one implicit step of several independent grids
    unet_forward  one apply of the learned preconditioner's network
    unet_grad     loss and weight gradient of one training pair
"""
import math

import numpy as np
import torch
import torch.nn.functional as nnf

from paper_2007_10411_gb300 import jfnk, synth

PRECOND = {"none": synth.PC_NONE, "block": synth.PC_BLOCK, "schur": synth.PC_SCHUR, "nonlinear": synth.PC_NONLINEAR}
CLOSURE = {"constant": synth.SGS_CONST, "smagorinsky": synth.SGS_SMAGORINSKY, "deardorff": synth.SGS_DEARDORFF}


def _step(problem, nx, nz, ny=0, precision="mixed", closure="smagorinsky", precond="block", sweeps=2, krylov=30):
    return {"kind": "step", "problem": problem, "nx": nx, "ny": ny, "nz": nz, "precision": precision,
            "closure": closure, "precond": precond, "sweeps": sweeps, "krylov": krylov}


def _operators(nx, nz, ny=0, closure="smagorinsky"):
    return {"kind": "operators", "problem": "thermal", "nx": nx, "ny": ny, "nz": nz, "precision": "fp64",
            "closure": closure, "precond": "block", "sweeps": 2, "krylov": 4}


def _unet(kind, nx, nz, ny=0):
    return {"kind": kind, "problem": "thermal", "nx": nx, "ny": ny, "nz": nz, "precision": "mixed",
            "closure": "smagorinsky", "precond": "block", "sweeps": 2, "krylov": 4}


def listed():
    return [
        # a small monitoring call: latency and launches count
        dict(_operators(100, 37), name="operators_100x37"),
        # the same call on a ragged 3-D grid
        dict(_operators(130, 45, ny=77, closure="deardorff"), name="operators_130x77x45"),
        # the smallest configuration: neutral thermal, constant coefficients, all float64
        dict(_step("thermal", 128, 64, precision="fp64", closure="constant"), name="step_fp64_128x64"),
        # a grid whose rows are neither a multiple of a tile nor of a vector load
        dict(_step("thermal", 250, 119), name="step_mixed_250x119"),
        # the benchmark workload: stable thermal, mixed precision, field-block preconditioner
        dict(_step("thermal", 1024, 512), name="step_mixed_1024x512"),
        # the same workload as the paper has it, all float64
        dict(_step("thermal", 1024, 512, precision="fp64"), name="step_fp64_1024x512"),
        # the fastest way to take that step: acoustic Schur complement
        dict(_step("thermal", 1024, 512, precond="schur", sweeps=32), name="step_schur_1024x512"),
        # sixteen heat islands of uneven sizes stepped together (no-slip ground, surface flux)
        dict(_step("heat_island", 512, 128, precond="schur", sweeps=16), kind="batch", n=16, name="batch16_heat_island"),
        # 3-D thermal, field block, FGMRES(20)
        dict(_step("thermal", 256, 64, ny=256, krylov=20), name="step3d_mixed_256x256x64"),
        # the largest 3-D thermal, Schur complement
        dict(_step("thermal", 256, 128, ny=256, precond="schur", sweeps=16, krylov=20), name="step3d_schur_256x256x128"),
        # learned preconditioner: one apply on the benchmark grid
        dict(_unet("unet_forward", 1024, 512), name="unet_forward_1024x512"),
        # learned preconditioner: one training pair's gradient
        dict(_unet("unet_grad", 256, 128), name="unet_grad_256x128"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["operators", "operators3d", "block", "block", "block64", "schur", "block3d", "schur3d", "batch",
                       "unet_forward", "unet_grad", "unet_forward3d"])
    closure = rng.choice(["constant", "smagorinsky", "smagorinsky", "smagorinsky", "deardorff"])
    problem = rng.choice(["thermal", "thermal", "heat_island"])
    if kind == "operators":
        return _operators(_log_int(rng, 48, 1500), _log_int(rng, 24, 700), closure=closure)
    if kind == "operators3d":
        return _operators(_log_int(rng, 24, 280), _log_int(rng, 12, 110), ny=_log_int(rng, 24, 200), closure=closure)
    if kind == "block":
        return _step("thermal", _log_int(rng, 48, 1030), _log_int(rng, 24, 500), closure=closure,
                     precond=rng.choice(["block", "block", "block", "nonlinear"]), sweeps=rng.choice([2, 2, 2, 3, 4]),
                     krylov=rng.choice([20, 30, 30]))
    if kind == "block64":
        return _step("thermal", _log_int(rng, 48, 400), _log_int(rng, 24, 260), precision="fp64", closure=closure)
    if kind == "schur":
        return _step(problem, _log_int(rng, 64, 1500), _log_int(rng, 32, 520), closure=closure, precond="schur",
                     sweeps=rng.choice([8, 16, 16, 24, 32, 33]), precision=rng.choice(["mixed", "mixed", "mixed", "fp64"]))
    if kind == "block3d":
        return _step("thermal", _log_int(rng, 30, 200), _log_int(rng, 16, 72), ny=_log_int(rng, 30, 200),
                     closure=closure, sweeps=rng.choice([2, 2, 3]), krylov=20)
    if kind == "schur3d":
        return _step(problem, _log_int(rng, 40, 256), _log_int(rng, 24, 128), ny=_log_int(rng, 40, 256),
                     closure=closure, precond="schur", sweeps=rng.choice([8, 16, 17]), krylov=20)
    if kind == "batch":
        c = _step("heat_island", _log_int(rng, 200, 520), _log_int(rng, 64, 128), precond="schur",
                  sweeps=rng.choice([8, 16]))
        return dict(c, kind="batch", n=rng.randint(2, 9))
    if kind == "unet_forward3d":
        return _unet("unet_forward", 32 * rng.randint(1, 8), 4 * _log_int(rng, 2, 20), ny=64 * rng.randint(1, 3))
    return _unet(kind, 32 * _log_int(rng, 2, 32 if kind == "unet_forward" else 12),
                 32 * _log_int(rng, 1, 16 if kind == "unet_forward" else 8))


# ------------------------------------------------------------------ parameters
def _one(case, nx, ny, nz, h0=100.0):
    """The package's parameter dict of one grid of the case."""
    if case["problem"] == "heat_island":
        c = synth.case("uhi3d_%dx%dx%d" % (nx, ny, nz) if ny else "uhi_%dx%d" % (nx, nz))
        c["init"]["H0"] = h0
    else:
        c = synth.case("thermal3d_%dx%dx%d" % (nx, ny, nz) if ny else "thermal_stable_%dx%d" % (nx, nz))
    if case["closure"] == "constant":
        c["sgs"].update(mode=synth.SGS_CONST)
        if case["problem"] == "thermal":
            c["strat"]["beta"] = 0.0
    else:
        c["sgs"].update(mode=CLOSURE[case["closure"]])
    c["opts"].update(precision=synth.PREC_FP64 if case["precision"] == "fp64" else synth.PREC_MIXED,
                     precond=PRECOND[case["precond"]], pc_sweeps=case["sweeps"], krylov_m=case["krylov"])
    return c


def _params(case):
    """One parameter dict per grid: heat islands of a batch differ in size and surface flux."""
    if case["kind"] != "batch":
        return [_one(case, case["nx"], case["ny"], case["nz"])]
    n = case["n"]
    return [_one(case, case["nx"] * (1 + i % 4), 0, case["nz"] * (1 + i // 8), 25.0 * (930.0 / 25.0) ** (i / max(n - 1, 1)))
            for i in range(n)]


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _state(c, seed):
    """A developed flow: divergence-free rolls, a warm bubble or surface layer, white noise on theta."""
    g, no_slip = c["grid"], c["grid"]["bc_bottom"] == synth.NOSLIP
    rng = np.random.default_rng(int(seed))
    kw = {"dtype": torch.float64, "device": "cuda"}
    three = g["dim"] == 3
    xs = (torch.arange(g["nx"], **kw) / g["nx"]).view(1, 1, -1)
    ys = (torch.arange(g["ny"], **kw) / g["ny"]).view(1, -1, 1) if three else torch.zeros(1, 1, 1, **kw)
    zs = ((torch.arange(g["nz"], **kw) + 0.5) / g["nz"]).view(-1, 1, 1)
    u = torch.zeros(synth.shape(c), **kw)
    full = u if three else u.unsqueeze(2)                       # [field][z][y][x]
    wind = 2.0 if no_slip else 4.0
    iw, it = (2, 3) if three else (1, 2)
    for axis, pos, length in ((0, xs, g["lx"]), (1, ys, g["ly"]))[: 2 if three else 1]:
        for m in (1, 2, 3):
            k, ph = 2 * math.pi * m, 2 * math.pi * rng.random()
            amp = wind * (0.5 + rng.random()) / m
            # psi = amp * lz / pi * s(z) * cos(k x + ph); s and, over a no-slip ground, s' vanish at the walls
            s, ds = (torch.sin(math.pi * zs) ** 2, torch.sin(2 * math.pi * zs)) if no_slip else \
                    (torch.sin(math.pi * zs), torch.cos(math.pi * zs))
            full[axis] += amp * ds * torch.cos(k * pos + ph)
            full[iw] += amp * (g["lz"] / math.pi) * s * (k / length) * torch.sin(k * pos + ph)
    noise = torch.randn(full[it].shape, generator=_gen(seed + 77), **kw)
    if no_slip:
        full[it] += 0.5 * torch.exp(-zs * g["lz"] / 200.0) * torch.exp(-((xs - 0.4 - 0.2 * rng.random()) / 0.1) ** 2) + 1e-3 * noise
    else:
        x0 = 0.35 + 0.3 * rng.random()
        r2 = ((xs - x0) * g["lx"] / 2000.0) ** 2 + ((zs * g["lz"] - 2000.0 - 1500.0 * rng.random()) / 2000.0) ** 2
        if three:
            r2 = r2 + ((ys - 0.35 - 0.3 * rng.random()) * g["ly"] / 2000.0) ** 2
        full[it] += 2.0 * torch.cos(0.5 * math.pi * torch.sqrt(r2).clamp(max=1.0)) ** 2 + 0.01 * noise
    return u.contiguous()


def _flux(c):
    if c["init"]["kind"] != "rest":
        return None
    return torch.from_numpy(np.ascontiguousarray(synth.heat_flux(c))).to("cuda", torch.float64)


#: network layers (name, inputs, outputs, kernel size), the flat weight order of the library
LAYERS = (("L0a", 16, 16, 3), ("L0b", 16, 16, 3), ("L1a", 16, 32, 3), ("L1b", 32, 32, 3), ("L2a", 32, 64, 3),
          ("L2b", 64, 64, 3), ("L1c", 96, 32, 3), ("L0c", 48, 16, 3), ("L0d", 16, 16, 1))


def _weights(seed):
    rng = np.random.default_rng(int(seed) + 5)
    return np.concatenate([rng.standard_normal(k * k * co * ci) / math.sqrt(k * k * ci) for _, ci, co, k in LAYERS]).astype(np.float32)


def _pair(c, seed):
    """A unit Krylov vector (a smooth part and noise in every field) and a target for it."""
    g = _gen(seed + 3)
    x = torch.randn(synth.shape(c), generator=g, device="cuda", dtype=torch.float32)
    u = _state(c, seed + 1).float()
    x = x + 2.0 * u / u.flatten(1).std(1).clamp(min=1e-6).view(-1, *[1] * (u.dim() - 1))
    t = torch.randn(x.shape, generator=g, device="cuda", dtype=torch.float32) + 0.5 * x
    return (x / x.norm()).contiguous(), (t / t.norm()).contiguous()


# ------------------------------------------------------------------ the library's calls
def prepare(case, seed):
    cs = _params(case)
    kind = case["kind"]
    if kind == "batch":
        u0 = [_state(c, seed + 1000 * i) for i, c in enumerate(cs)]
        b = jfnk.Batch(cs)
        for i, c in enumerate(cs):
            b.set_surface_flux(i, _flux(c))
        return {"kind": kind, "solver": b, "u0": u0, "u": [torch.empty_like(u) for u in u0]}
    c = cs[0]
    s = jfnk.Solver(c)
    if kind.startswith("unet"):
        s.unet_init(0)
        s.unet_set_weights(_weights(seed))
        x, t = _pair(c, seed)
        return {"kind": kind, "solver": s, "x": x, "t": t, "y": torch.empty_like(x)}
    H = _flux(c)
    if H is not None:
        s.set_surface_flux(H)
    u0 = _state(c, seed)
    st = {"kind": kind, "solver": s, "u0": u0, "u": torch.empty_like(u0)}
    if kind == "operators":
        st["u"] = u0 + 0.1 * _state(c, seed + 500)
        st["F"], st["R"] = torch.empty_like(u0), torch.empty_like(u0)
    return st


def run(s):
    kind, solver = s["kind"], s["solver"]
    if kind == "operators":
        solver.rhs(s["u"], s["F"])
        solver.residual(s["u0"], s["u"], s["R"])
        return {"F": s["F"], "R": s["R"]}
    if kind == "unet_forward":
        solver.unet_forward(s["x"], s["y"])
        return s["y"]
    if kind == "unet_grad":
        loss, grad = solver.unet_loss_grad(s["x"], s["t"])
        return {"loss": loss, "grad": grad}
    if kind == "batch":
        for u, u0 in zip(s["u"], s["u0"]):       # the program keeps u^n
            u.copy_(u0)
        solver.step(s["u"])
        return s["u"]
    s["u"].copy_(s["u0"])
    solver.step(s["u"])
    return s["u"]


def work(case):
    """State (or operand) bytes in and out once; F costs about 130 (2-D) / 230 (3-D) operations a point."""
    flops = nbytes = 0.0
    for c in _params(case):
        g = c["grid"]
        npt = g["nx"] * g["nz"] * (g["ny"] if g["dim"] == 3 else 1)
        n, f = npt * synth.n_fields(c), npt * (230.0 if g["dim"] == 3 else 130.0)
        if case["kind"] == "operators":
            nbytes, flops = nbytes + 8.0 * 4 * n, flops + 3 * f          # u^n, u in; F, R out
        elif case["kind"].startswith("unet"):
            per = 32128.0 if g["dim"] == 3 else 47360.0                   # operations of all layers, per point
            back = case["kind"] == "unet_grad"
            nbytes, flops = nbytes + 4.0 * 2 * n, flops + per * npt * (3.0 if back else 1.0)
        else:
            # u^n in, u^{n+1} out; at least two Newton corrections, each a residual and a Jacobian product
            nbytes, flops = nbytes + 8.0 * 2 * n, flops + 5 * f
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------ 64-bit results
class _Model:
    """F(u) of the semi-discrete equations on [field][z][y][x] (2-D: one y), float64."""

    def __init__(self, c, heat):
        g, s, q, o = c["grid"], c["strat"], c["sgs"], c["opts"]
        self.three = g["dim"] == 3
        self.s, self.q, self.dt = s, q, o["dt"]
        self.h = {-1: g["lx"] / g["nx"], -2: g["ly"] / g["ny"] if self.three else 1.0, -3: g["lz"] / g["nz"]}
        nf = 5 if self.three else 4
        self.vel = [-1, -2, -3] if self.three else [-1, -3]          # axis of each velocity component
        self.iw, self.it, self.ip = nf - 3, nf - 2, nf - 1
        hor = [1.0 if g["bc_bottom"] == synth.FREESLIP else -1.0, 1.0 if g["bc_top"] == synth.FREESLIP else -1.0]
        self.par = [hor] * (nf - 3) + [[-1.0, -1.0], [1.0, 1.0], [1.0, 1.0]]
        sc = [o["scale_u"]] * (nf - 2) + [o["scale_theta"], o["scale_p"]]
        self.scale = torch.tensor(sc, dtype=torch.float64, device="cuda").view(-1, 1, 1, 1)
        self.heat = None
        if heat is not None:
            self.heat = torch.zeros(g["nz"], g["ny"] if self.three else 1, g["nx"], dtype=torch.float64, device="cuda")
            self.heat[0] = heat.view(self.heat[0].shape) / (s["rho0"] * s["cp"] * self.h[-3])

    def d(self, f, axis, par=(1.0, 1.0)):
        if axis != -3:
            r = lambda k: torch.roll(f, -k, axis)  # noqa: E731
            return (2 / 3 * (r(1) - r(-1)) - 1 / 12 * (r(2) - r(-2))) / self.h[axis]
        n = f.shape[0]
        e = torch.cat([par[0] * f[:2].flip(0), f, par[1] * f[-2:].flip(0)])
        return (2 / 3 * (e[3:n + 3] - e[1:n + 1]) - 1 / 12 * (e[4:n + 4] - e[0:n])) / self.h[-3]

    def closure(self, grads):
        """(K for momentum, K for heat) by axis."""
        q, s = self.q, self.s
        if q["mode"] == synth.SGS_CONST:
            return {a: (q["K_M"], q["K_H"]) for a in self.vel}
        ss = 0.0
        for i, a in enumerate(self.vel):
            for j, b in enumerate(self.vel):
                ss = ss + (0.5 * (grads[i][b] + grads[j][a])) ** 2
        dx, dz = self.h[-1], self.h[-3]
        dy = self.h[-2] if self.three else dx
        delta = (dx * dy * dz) ** (1 / 3) if self.three else math.sqrt(dx * dz)
        st = torch.sqrt(2 * ss + 1e-300)
        nu = (q["Cs"] * delta) ** 2 * st
        if q["mode"] == synth.SGS_SMAGORINSKY:
            return {a: (nu, nu / q["Pr"]) for a in self.vel}
        # eps = nu S:S with S:S = s^2 / 2, so eps^(1/3) = ((Cs delta)^2 / 2)^(1/3) s
        base = q["Cs"] ** (4 / 3) * (0.5 * (q["Cs"] * delta) ** 2) ** (1 / 3) * st
        n2 = s["g"] * s["beta"] / s["theta0"]
        ml = torch.clamp(0.75 * nu / (0.1 * delta) / math.sqrt(n2), max=delta) if n2 > 0 else delta
        km, kM = base * (dx * dy) ** (2 / 3), base * dz ** (4 / 3)
        hor = (km, km * (1 + 2 * ml / math.sqrt(dx * dy)))
        return {a: hor if a != -3 else (kM, kM * (1 + 2 * ml / dz)) for a in self.vel}

    def F(self, u):
        s, out = self.s, []
        grads = [{a: self.d(u[f], a, self.par[f]) for a in self.vel} for f in range(len(u))]
        K = self.closure(grads)
        div = sum(grads[i][a] for i, a in enumerate(self.vel))
        for f in range(len(u)):
            r = 0.0
            for i, a in enumerate(self.vel):
                pp = [self.par[f][k] * self.par[self.iw][k] for k in (0, 1)]
                r = r - 0.5 * self.d(u[i] * u[f], a, pp) - 0.5 * u[i] * grads[f][a]
                if f != self.ip:
                    k = K[a][1 if f == self.it else 0]
                    r = r + self.d(k * grads[f][a], a, [-self.par[f][0], -self.par[f][1]])
            if f <= self.iw:
                r = r - s["theta0"] * grads[self.ip][self.vel[f]]
            if f == self.iw:
                r = r + s["g"] / s["theta0"] * u[self.it]
            if f == self.it:
                r = r - s["beta"] * u[self.iw]
                if self.heat is not None:
                    r = r + self.heat
            if f == self.ip:
                r = r - s["gamma_p"] * (s["pbar"] + u[f]) * div
            out.append(r)
        return torch.stack(out)

    def wave_solve(self, r):
        """(2/dt + acoustic terms)^-1 r on the mirror-extended periodic box (a preconditioner)."""
        nz = r.shape[1]
        half = self.dt / 2
        even = [-1.0 if f == self.iw else 1.0 for f in range(len(r))]
        ext = torch.stack([torch.cat([r[f], even[f] * r[f].flip(0)]) for f in range(len(r))])
        hat = torch.fft.fftn(ext, dim=(-3, -2, -1))
        sym = {}
        for a in self.vel:
            n = ext.shape[a]
            t = 2 * math.pi * torch.fft.fftfreq(n, dtype=torch.float64, device="cuda")
            shape = [1, 1, 1]
            shape[a] = n
            sym[a] = ((4 / 3 * torch.sin(t) - 1 / 6 * torch.sin(2 * t)) / self.h[a]).view(shape)
        k2 = sum(v ** 2 for v in sym.values())
        cg, th = self.s["gamma_p"] * self.s["pbar"], self.s["theta0"]
        kr = sum(1j * sym[a] * hat[i] for i, a in enumerate(self.vel))
        p = (hat[self.ip] - cg * half * kr) / (2 / self.dt + cg * th * half * k2)
        sol = [half * (hat[i] - th * 1j * sym[a] * p) for i, a in enumerate(self.vel)] + [half * hat[self.it], p]
        return torch.fft.ifftn(torch.stack(sol), dim=(-3, -2, -1)).real[:, :nz].contiguous()


def _gmres(A, M, b, tol, m=25, cycles=6):
    x = torch.zeros_like(b)
    r, stop = b, tol * b.norm()
    for _ in range(cycles):
        beta = r.norm()
        if beta <= stop:
            break
        V, Z, H = [r / beta], [], torch.zeros(m + 1, m, dtype=torch.float64)
        for j in range(m):
            Z.append(M(V[j]))
            w = A(Z[j])
            for _again in (0, 1):
                for i in range(j + 1):
                    hij = (V[i] * w).sum()
                    H[i, j] += float(hij)
                    w = w - hij * V[i]
            H[j + 1, j] = float(w.norm())
            e = torch.zeros(j + 2, dtype=torch.float64)
            e[0] = float(beta)
            y = torch.linalg.lstsq(H[: j + 2, : j + 1], e).solution
            if float((e - H[: j + 2, : j + 1] @ y).norm()) <= float(stop) or float(H[j + 1, j]) == 0.0:
                break
            V.append(w / float(H[j + 1, j]))
        for yi, zi in zip(y.tolist(), Z):
            x = x + yi * zi
        r = b - A(x)
    return x


def _exact_step(c, u0):
    m = _Model(c, _flux(c))
    un = u0.view(len(u0), c["grid"]["nz"], -1, c["grid"]["nx"])
    two, W = 2.0 / m.dt, m.scale
    f = two * un + m.F(un)
    u, first = un, None
    for _ in range(8):
        R = two * u - m.F(u) - f
        norm = float((R / W).norm())
        first = first or norm
        if norm <= 1e-13 * first:
            break
        jac = lambda v: (two * W * v - torch.func.jvp(m.F, (u,), (W * v,))[1]) / W  # noqa: E731,B023
        step = _gmres(jac, lambda v: m.wave_solve(W * v) / W, -R / W, 1e-7)
        u = u + W * step
        if float(step.norm()) <= 1e-15 * float((u / W).norm()):
            break
    return u.reshape(u0.shape).contiguous()


def _exact_net(c, w, x):
    """N(x) = B^-1 net(B x) in float64; x [field][z][x] or [field][z][y][x]."""
    s, o, three = c["strat"], c["opts"], c["grid"]["dim"] == 3
    bal = torch.ones(len(x), dtype=torch.float64, device="cuda")
    if s["beta"] != 0.0:
        bal[-2] = o["scale_theta"] / (o["scale_u"] * math.sqrt(abs(s["beta"]) * s["theta0"] / s["g"]))
    bal[-1] = o["scale_p"] / (o["scale_u"] * math.sqrt(s["gamma_p"] * s["pbar"] / s["theta0"]))
    bal = bal.view(-1, *[1] * (x.dim() - 1))
    ws, at = {}, 0
    for name, ci, co, k in LAYERS:
        ws[name] = w[at:at + k * k * co * ci].view(k, k, co, ci).permute(2, 3, 0, 1)
        at += k * k * co * ci

    def conv(name, a):                                   # a: [plane][channel][row][column]
        return nnf.conv2d(a, ws[name], padding=ws[name].shape[-1] // 2)

    def pool(a):
        a = nnf.avg_pool2d(a, 2)
        return 0.5 * (a[0::2] + a[1::2]) if three else a

    def up(a):
        a = a.repeat_interleave(2, -1).repeat_interleave(2, -2)
        return a.repeat_interleave(2, 0) if three else a

    a = bal * x
    a = a.transpose(0, 1) if three else a.unsqueeze(0)
    a = torch.cat([a, a.new_zeros(a.shape[0], 16 - a.shape[1], *a.shape[2:])], 1)
    s0 = conv("L0b", conv("L0a", a))
    s1 = conv("L1b", conv("L1a", pool(s0)))
    b2 = conv("L2b", conv("L2a", pool(s1)))
    c1 = conv("L1c", torch.cat([up(b2), s1], 1))
    y = conv("L0d", conv("L0c", torch.cat([up(c1), s0], 1)))[:, : len(x)]
    return (y.transpose(0, 1) if three else y[0]) / bal, bal


def exact(case, seed):
    cs, kind = _params(case), case["kind"]
    if kind == "batch":
        return [_exact_step(c, _state(c, seed + 1000 * i)) for i, c in enumerate(cs)]
    c = cs[0]
    if kind == "step":
        return _exact_step(c, _state(c, seed))
    if kind == "operators":
        m, g = _Model(c, _flux(c)), c["grid"]
        u0 = _state(c, seed)
        u = u0 + 0.1 * _state(c, seed + 500)
        v0, v = (a.view(len(a), g["nz"], -1, g["nx"]) for a in (u0, u))
        F, two = m.F(v), 2.0 / m.dt
        return {"F": F.reshape(u.shape), "R": (two * v - F - two * v0 - m.F(v0)).reshape(u.shape)}
    x, t = _pair(c, seed)
    w = torch.from_numpy(_weights(seed)).to("cuda", torch.float64)
    if kind == "unet_forward":
        return _exact_net(c, w, x.double())[0].contiguous()
    w.requires_grad_(True)
    y, bal = _exact_net(c, w, x.double())
    loss = 0.5 * ((bal * (y - t.double())) ** 2).sum() / ((bal * x.double()) ** 2).sum()
    grad = torch.autograd.grad(loss, w)[0]
    return {"loss": float(loss.detach()), "grad": grad}
