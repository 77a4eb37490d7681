"""The workloads this solver is timed on, each through the package's public calls.

Four kinds of work, over the sizes of the presets in lbpc_inputs.py, of bench.py and of the
tests:

  run      advance a lattice by a block of steps and read its fields;
  monitor  the same with dense in-run diagnostics and the scalars read at the end;
  restart  load a state from device arrays, advance it, and read the populations back;
  adjoint  one evaluation of the liquid volume and its gradients (fresh lattice, forward,
           backward), as an optimisation of the wall temperature calls it.

States are those of a run under way: a melted layer behind a wavy front, a convection roll in
the liquid, solid at the melting temperature with the usual tiny perturbation ahead of it.
Fields are handed on in the precision the lattice computes in (FP64 storage: float64, every
other mode: float32), as a program that goes on to plot or store them does.
"""
from __future__ import annotations

import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

import lbpc_inputs as inp
from paper_1703_02652_gb300 import LBPC, liquid_volume

STORAGE = {"f64": inp.FP64, "f32": inp.FP32, "f16": inp.FP16, "bf16": inp.BF16,
           "f16g32": inp.FP16_G32, "bf16g32": inp.BF16_G32}
F_BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2, "f16g32": 2, "bf16g32": 2}
G_BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2, "f16g32": 4, "bf16g32": 4}
#: node updates of a pass: the largest listed case, with room below it for the slower options
MOST_UPDATES = 256 ** 3 * 50


def _case(kind, nx, ny, nz, storage, steps, **kw):
    """A case with every option spelled out.  walls: "cavity" (hot and cold x walls, the other
    faces adiabatic), "slab" (the same, periodic along y) or "column" (hot x wall, adiabatic
    far wall, periodic along y and z)."""
    c = dict(kind=kind, nx=nx, ny=ny, nz=nz, storage=storage, steps=steps, flow="mrt",
             enthalpy="mrt", walls="cavity", aa=False, Ra=1e6, Pr=0.02, St=1.0, tau_g=0.0,
             report_every=500, ckpt_every=0)
    c.update(kw)
    return c


def listed():
    def named(name, c):
        return dict(name=name, **c)

    return [
        # the 1D melting run against the Neumann solution, the smallest lattice in use
        named("stefan_64x4x4_f64", _case("run", 64, 4, 4, "f64", 200, flow="none", walls="column",
                                         tau_g=0.8, St=0.1, report_every=0)),
        # 2D conduction on the corner-solidification grid
        named("plane_128x1x128_f64", _case("run", 128, 1, 128, "f64", 100, flow="none",
                                           walls="slab", tau_g=0.9, St=1.2, report_every=0)),
        # quasi-2D convective melting: many steps on a small plane
        named("melting2d_64x1x64_f32", _case("run", 64, 1, 64, "f32", 200, walls="slab", Ra=2.5e4,
                                             St=0.01, report_every=0)),
        # the 64^3 cavity, whose state stays in the L2
        named("cavity_64_f32", _case("run", 64, 64, 64, "f32", 100, Ra=1e5)),
        # FP64 storage: the reference trajectory of a precision study
        named("cavity_128_f64", _case("run", 128, 128, 128, "f64", 10)),
        # odd extents: a grid with a node on the mid-planes
        named("cavity_161x161x81_f32", _case("run", 161, 161, 81, "f32", 50)),
        # the headline lattice in the storage and streaming options of production runs
        named("cavity_256_f32", _case("run", 256, 256, 256, "f32", 50)),
        named("cavity_256_f16", _case("run", 256, 256, 256, "f16", 50, Pr=50.0)),
        named("cavity_256_f16_aa", _case("run", 256, 256, 256, "f16", 50, aa=True, Pr=50.0)),
        # a production grid with its Nusselt number and front recorded every ten steps
        named("monitor_160x160x80_f16g32", _case("monitor", 160, 160, 80, "f16g32", 50,
                                                 report_every=10)),
        # resume from populations held on the device and hand them on again
        named("restart_128_bf16", _case("restart", 128, 128, 128, "bf16", 10, Pr=6.2)),
        # gradient of the liquid volume with respect to the wall temperature and St
        named("adjoint_96_f32", _case("adjoint", 96, 96, 96, "f32", 200, Ra=1e5, Pr=6.2,
                                      report_every=0, ckpt_every=50)),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["run", "run", "run", "run", "monitor", "restart", "adjoint"])
    storage = rng.choice(["f64", "f32", "f32", "f16", "f16", "bf16", "f16g32", "bf16g32"])
    flow = rng.choice(["mrt", "mrt", "mrt", "srt", "none"])
    walls = rng.choice(["cavity", "cavity", "slab"]) if flow != "none" else rng.choice(
        ["cavity", "slab", "column"])
    nx = log(24, 256)
    ny = 1 if walls == "slab" and rng.random() < 0.5 else log(4, min(256, 2 * nx))
    nz = log(4, min(256, 2 * nx))
    if rng.random() < 0.5:
        nx += nx % 2
    most = MOST_UPDATES // (24 if storage == "f64" and flow != "none" else 2)
    if kind == "adjoint":
        storage = rng.choice(["f32", "f32", "f16"])
        nx, ny, nz = min(nx, 96), min(ny, 96), min(nz, 96)
        steps = rng.choice([50, 100, 150])
        return _case(kind, nx, ny, nz, storage, steps, flow="mrt", walls="cavity", Ra=1e5, Pr=6.2,
                     report_every=0, ckpt_every=rng.choice([25, 40, 50]))
    steps = max(4, min(log(10, 200), most // (nx * ny * nz)))
    report = rng.choice([0, 500, 500]) if kind != "monitor" else rng.choice([5, 10, 25])
    kw = dict(Ra=rng.choice([1e5, 1e6]), Pr=rng.choice([0.02, 6.2, 50.0]))
    if nx < 64:  # what so coarse a grid resolves
        kw["Ra"] = 1e4
    if storage in ("f16", "bf16"):
        kw["Pr"] = rng.choice([6.2, 50.0])
    if flow == "srt":
        kw["Pr"] = 6.2
    if flow == "none":
        kw = dict(tau_g=round(rng.uniform(0.6, 1.2), 3), St=rng.choice([0.1, 1.0]))
    return _case(kind, nx, ny, nz, storage, steps, flow=flow, walls=walls,
                 enthalpy=rng.choice(["mrt", "mrt", "srt"]), report_every=report,
                 aa=kind != "restart" and rng.random() < 0.3, **kw)


def _params(c):
    far = inp.ADIABATIC if c["walls"] == "column" else inp.ISOTHERMAL
    y = inp.ADIABATIC if c["walls"] == "cavity" else inp.PERIODIC
    z = inp.PERIODIC if c["walls"] == "column" else inp.ADIABATIC
    return inp.Params(
        flow_model={"none": inp.FLOW_NONE, "mrt": inp.FLOW_MRT, "srt": inp.FLOW_SRT}[c["flow"]],
        enth_model={"mrt": inp.ENTH_MRT, "srt": inp.ENTH_SRT}[c["enthalpy"]],
        precision=STORAGE[c["storage"]], streaming=inp.AA if c["aa"] else inp.PULL,
        bc=[inp.ISOTHERMAL, far, y, y, z, z], Ra=c["Ra"], Pr=c["Pr"], St=c["St"],
        tau_g=c["tau_g"], report_every=c["report_every"])


# ------------------------------------------------------------------------------------------
# States
# ------------------------------------------------------------------------------------------
def _velocities():
    """D3Q19 velocities: rest, the axis pairs, then the xy, xz and yz diagonals."""
    e = [(0, 0, 0)]
    for ax in range(3):
        for s in (1, -1):
            v = [0, 0, 0]
            v[ax] = s
            e.append(tuple(v))
    for a, b in ((0, 1), (0, 2), (1, 2)):
        for sb in (1, -1):
            for sa in (1, -1):
                v = [0, 0, 0]
                v[a], v[b] = sa, sb
                e.append(tuple(v))
    return e


E19 = _velocities()
W19 = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
OMEGA_T = 0.25


def _melted(c, seed):
    """(h, T, f_l, u) of a half-melted lattice, FP64 on the device, arrays (nz, ny, nx)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    r = np.random.default_rng(seed)
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    kw = dict(dtype=torch.float64, device="cuda")
    X = ((torch.arange(nx, **kw) + 0.5) / nx).view(1, 1, nx)
    Y = ((torch.arange(ny, **kw) + 0.5) / ny).view(1, ny, 1)
    Z = ((torch.arange(nz, **kw) + 0.5) / nz).view(nz, 1, 1)
    pi = math.pi
    front = r.uniform(0.35, 0.6) + r.uniform(0.03, 0.1) * torch.cos(
        2 * pi * Z + r.uniform(0, 6)) * (1 + 0.3 * torch.cos(2 * pi * Y + r.uniform(0, 6)))
    fl = torch.clamp((front - X) * nx / 1.5 + 0.5, 0.0, 1.0)
    noise = torch.rand((nz, ny, nx), generator=gen, **kw) * 2 - 1
    liquid = fl >= 1
    T = torch.where(liquid, torch.clamp((1 - X / front) * (1 + 2e-3 * noise), min=0.0),
                    torch.where(fl > 0, 0.0, torch.clamp(1e-6 * noise, max=0.0)))
    latent = 1.0 / c["St"]
    h = T + latent * fl + torch.where(fl > 0, 0.0, torch.clamp(1e-6 * noise, min=0.0))
    fl = torch.clamp(h / latent, 0.0, 1.0)
    a = pi / front
    inside = (X < front) * r.uniform(0.008, 0.02)
    sx, sz = torch.sin(a * X), torch.sin(pi * Z)
    u = torch.stack([-inside * sx * sx * 2 * sz * torch.cos(pi * Z),
                     0.1 * inside * sx * sz * torch.sin(2 * pi * Y),
                     inside * 2 * sx * torch.cos(a * X) * sz * sz]) * (fl >= 1)
    return h, T, fl, u


def _populations(c, seed):
    """(f or None, g): equilibrium populations of the melted state, (19, N) and (7, N)."""
    h, T, fl, u = _melted(c, seed)
    f = None
    if c["flow"] == "none":
        u = torch.zeros_like(u)
    else:
        f = torch.empty((19,) + tuple(h.shape), dtype=torch.float64, device="cuda")
        u2 = (u * u).sum(0)
        rho = 1 + 1e-3 * (T - 0.3) * (fl >= 1)
        for q, (e, w) in enumerate(zip(E19, W19)):
            eu = e[0] * u[0] + e[1] * u[1] + e[2] * u[2]
            f[q] = w * (rho + 3 * eu + 4.5 * eu * eu - 1.5 * u2)
        f = f.view(19, -1)
    g = torch.empty((7,) + tuple(h.shape), dtype=torch.float64, device="cuda")
    for ax in range(3):
        for s in (0, 1):
            g[1 + 2 * ax + s] = 0.5 * OMEGA_T * T + (0.5 - s) * T * u[ax]
    g[0] = h - g[1:].sum(0)
    return f, g.view(7, -1)


def _wall(c, seed):
    """Hot-wall temperature field of the adjoint, 1 + 0.05 N(0, 1), float32 on the device."""
    T = inp.wall_temperature_field(c["ny"], c["nz"], seed=seed)
    return torch.from_numpy(T).float().cuda()


def prepare(case, seed):
    shape, p = (case["nx"], case["ny"], case["nz"]), _params(case)
    if case["kind"] == "adjoint":
        h0 = _melted(case, seed)[0].reshape(-1).cpu().numpy()
        return {"case": case, "shape": shape, "params": p, "h0": h0, "T_wall": _wall(case, seed)}
    f, g = _populations(case, seed)
    lat = LBPC(shape, p)
    lat.set_distributions(f, g)
    state = {"case": case, "lat": lat}
    if case["kind"] == "restart":
        state.update(f=f, g=g)
    return state


def run(state):
    c = state["case"]
    if c["kind"] == "adjoint":
        Tw = state["T_wall"].detach().requires_grad_(True)
        St = torch.tensor(c["St"], dtype=torch.float64, requires_grad=True)
        J = liquid_volume(Tw, St, state["shape"], state["params"], state["h0"], c["steps"],
                          c["ckpt_every"])
        J.backward()
        return {"J": float(J), "dTw": Tw.grad, "dSt": float(St.grad)}
    lat = state["lat"]
    as_computed = torch.float64 if c["storage"] == "f64" else torch.float32
    if c["kind"] == "restart":
        lat.set_distributions(state["f"], state["g"])
        lat.step(c["steps"])
        f, g = lat.distributions()
        out = {"g": g.to(as_computed)}
        if f is not None:
            out["f"] = f.to(as_computed)
        return out
    lat.step(c["steps"])
    out = {k: v.to(as_computed) for k, v in lat.fields().items()}
    if c["flow"] == "none":
        del out["rho"], out["u"]  # zeros without a flow lattice
    if c["kind"] == "monitor":
        s = lat.scalars()
        out["scalars"] = {k: s[k] for k in ("liquid_vol", "nu_hot", "front_mean", "sum_h",
                                            "nu_fd", "front_mid")}
    return out


def work(case):
    """One read and one write of every stored population and of the FP64 rest channel per
    step; the outputs written once.  The adjoint: its forward, one reverse step per step on
    the 26 adjoint values, and the tape of 5 values written and read once."""
    n = case["nx"] * case["ny"] * case["nz"]
    flow = case["flow"] != "none"
    step = 2 * (19 * F_BYTES[case["storage"]] * flow + 6 * G_BYTES[case["storage"]] + 8)
    flops = 420 if flow else 70
    bytes_, ops = case["steps"] * step * n, case["steps"] * flops * n
    if case["kind"] == "adjoint":
        bytes_ += case["steps"] * (2 * 26 * 4 + 2 * 5 * 4) * n
        ops += case["steps"] * 600 * n
    elif case["kind"] == "restart":
        bytes_ += 2 * 8 * (19 * flow + 7) * n
    else:
        bytes_ += 8 * (7 if flow else 3) * n
    return {"bytes": float(bytes_), "flops": float(ops)}


# ------------------------------------------------------------------------------------------
# The same computations in plain FP64 tensors
# ------------------------------------------------------------------------------------------
def _moments19():
    """Rows of the orthogonal D3Q19 moment basis, and their squared norms."""
    e = np.array(E19, dtype=np.float64)
    x, y, z = e.T
    s = (e * e).sum(1)
    rows = [np.ones(19), 19 * s - 30, (21 * s * s - 53 * s + 24) / 2]
    for v in (x, y, z):
        rows += [v, (5 * s - 9) * v]
    a, b = 3 * x * x - s, y * y - z * z
    rows += [a, (3 * s - 5) * a, b, (3 * s - 5) * b, x * y, y * z, x * z,
             (y * y - z * z) * x, (z * z - x * x) * y, (x * x - y * y) * z]
    M = np.array(rows)
    return M, (M * M).sum(1)


class _Plain:
    """The coupled step on (19 | 7, nz, ny, nx) FP64 tensors: dense moment matrices, streaming
    by shifted copies with the half-way wall rules."""

    def __init__(self, c):
        self.c = c
        H, dT = float(c["nx"]), 1.0
        if c["flow"] != "none":
            U0 = 0.1 / math.sqrt(3.0)
            nu = U0 * H * math.sqrt(c["Pr"] / c["Ra"])
            chi = nu / c["Pr"]
            self.gbeta = U0 * U0 / (dT * H)
            s_nu = 1 / (3 * nu + 0.5)
            rate = {"e": 1.19, "eps": 1.4, "q": 1.2, "pi": 1.4, "t": 1.98, "nu": s_nu}
            if c["flow"] == "srt":
                rate = {k: s_nu for k in rate}
            order = ["", "e", "eps", "", "q", "", "q", "", "q", "nu", "pi", "nu", "pi", "nu", "nu",
                     "nu", "t", "t", "t"]
            self.S = self.column([rate.get(k, 0.0) for k in order])
            M, norm = _moments19()
            self.M = torch.tensor(M, device="cuda")
            self.Mi = torch.tensor((M / norm[:, None]).T.copy(), device="cuda")
        if c["tau_g"] > 0:
            chi = (c["tau_g"] - 0.5) * OMEGA_T
        s_chi = 1 / (chi / OMEGA_T + 0.5)
        s4 = 2 - s_chi if c["enthalpy"] == "mrt" else s_chi
        N = np.zeros((7, 7))
        N[0] = 1
        for ax in range(3):
            N[1 + ax, 1 + 2 * ax], N[1 + ax, 2 + 2 * ax] = 1, -1
        N[4] = [6] + [-1] * 6
        N[5] = [0, 2, 2, -1, -1, -1, -1]
        N[6] = [0, 0, 0, 1, 1, -1, -1]
        R = np.diag([0, s_chi, s_chi, s_chi, s4, s4, s4])
        self.K = torch.tensor(np.linalg.inv(N) @ R @ N, device="cuda")
        bc = {"cavity": "iiaaaa", "slab": "iippaa", "column": "iapppp"}[c["walls"]]
        self.wall = [b != "p" for b in bc]
        self.iso = [b == "i" for b in bc]

    @staticmethod
    def column(v):
        return torch.tensor(v, dtype=torch.float64, device="cuda").view(-1, 1, 1, 1)

    @staticmethod
    def invert(h, latent):
        fl = torch.clamp(h / latent, 0.0, 1.0)
        T = torch.where(h <= 0, h, torch.where(h >= latent, h - latent, 0.0))
        return T, fl

    def macros(self, f, g, latent):
        h = g.sum(0)
        T, fl = self.invert(h, latent)
        if f is None:
            return h, T, fl, None, None, None
        e = torch.tensor(E19, dtype=torch.float64, device="cuda")
        rho = f.sum(0)
        j = (e.T @ f.reshape(19, -1)).reshape((3,) + tuple(h.shape))
        Fb = self.gbeta * (T - 0.5)
        us = torch.stack([j[0], j[1], j[2] + 0.5 * Fb])
        F = -2 * (1 - fl) * us
        F = torch.stack([F[0], F[1], F[2] + Fb])
        return h, T, fl, rho, fl * us, F

    def collide(self, f, g, latent):
        h, T, fl, rho, u, F = self.macros(f, g, latent)
        if f is not None:
            ux, uy, uz = u
            Fx, Fy, Fz = F
            u2, Fu = (u * u).sum(0), (F * u).sum(0)
            zero = torch.zeros_like(rho)
            pxx, pww = 2 * ux * ux - uy * uy - uz * uz, uy * uy - uz * uz
            meq = rho * torch.stack([
                1 + zero, -11 + 19 * u2, 3 - 5.5 * u2, zero, -2 / 3 * ux, zero, -2 / 3 * uy, zero,
                -2 / 3 * uz, pxx, -0.5 * pxx, pww, -0.5 * pww, ux * uy, uy * uz, ux * uz, zero,
                zero, zero])
            a, b = 6 * Fx * ux - 2 * Fu, 2 * (Fy * uy - Fz * uz)
            FF = torch.stack([
                zero, 38 * Fu, -11 * Fu, Fx, -2 / 3 * Fx, Fy, -2 / 3 * Fy, Fz, -2 / 3 * Fz, a,
                -0.5 * a, b, -0.5 * b, Fx * uy + Fy * ux, Fy * uz + Fz * uy, Fx * uz + Fz * ux,
                zero, zero, zero])
            m = (self.M @ f.reshape(19, -1)).reshape(f.shape)
            # the conserved rows: the density as it is, the momentum raised by the force
            d = torch.where(self.S > 0, self.S * (meq - m), 0.0) + (1 - self.S / 2) * FF
            f = f + (self.Mi @ d.reshape(19, -1)).reshape(f.shape)
        eq = [None] * 7
        for ax in range(3):
            for s in (0, 1):
                v = 0.5 * OMEGA_T * T
                eq[1 + 2 * ax + s] = v if u is None else v + (0.5 - s) * T * u[ax]
        eq[0] = h - sum(eq[1:])
        d = g - torch.stack(eq)
        g = g - (self.K @ d.reshape(7, -1)).reshape(g.shape)
        return f, g

    def stream(self, p, vel, opp, Tw=None):
        """Pull of every population; behind a wall the node's own opposite one comes back
        (for g negated at an isothermal wall, plus its source)."""
        out = []
        for q, e in enumerate(vel):
            v = torch.roll(p[q], shifts=(e[2], e[1], e[0]), dims=(0, 1, 2)) if any(e) else p[q]
            for ax, dim in ((0, 2), (1, 1), (2, 0)):
                face = 2 * ax + (0 if e[ax] > 0 else 1)
                if e[ax] == 0 or not self.wall[face]:
                    continue
                n = v.shape[dim]
                back = p[opp[q]].narrow(dim, 0 if e[ax] > 0 else n - 1, 1)
                if Tw is not None and self.iso[face]:
                    back = -back + OMEGA_T * Tw[face]
                rest = v.narrow(dim, 1 if e[ax] > 0 else 0, n - 1)
                v = torch.cat([back, rest] if e[ax] > 0 else [rest, back], dim)
            out.append(v)
        return torch.stack(out)

    def step(self, f, g, latent, hot):
        f, g = self.collide(f, g, latent)
        if f is not None:
            opp = [E19.index(tuple(-a for a in e)) for e in E19]
            f = self.stream(f, E19, opp)
        g = self.stream(g, E19[:7], [0, 2, 1, 4, 3, 6, 5], [hot, 0.0, 0.0, 0.0, 0.0, 0.0])
        return f, g


def exact(case, seed):
    c, plain = case, _Plain(case)
    shape = (c["nz"], c["ny"], c["nx"])
    if c["kind"] == "adjoint":
        h = _melted(c, seed)[0]
        T = plain.invert(h, 1.0 / c["St"])[0]
        f = plain.column(W19).expand((19,) + shape).contiguous()
        g = torch.stack([h - 3 * OMEGA_T * T] + [0.5 * OMEGA_T * T] * 6)
        Tw = _wall(c, seed).double().requires_grad_(True)
        St = torch.tensor(c["St"], dtype=torch.float64, device="cuda", requires_grad=True)
        for _ in range(c["steps"]):
            f, g = checkpoint(lambda f, g, Tw, St: plain.step(f, g, 1.0 / St,
                                                              Tw.view(shape[0], shape[1], 1)),
                              f, g, Tw, St, use_reentrant=False)
        J = plain.invert(g.sum(0), 1.0 / St)[1].sum()
        J.backward()
        return {"J": float(J.detach()), "dTw": Tw.grad, "dSt": float(St.grad)}
    latent = 1.0 / c["St"]
    f, g = _populations(c, seed)
    f = f.view((19,) + shape) if f is not None else None
    g = g.view((7,) + shape)
    for _ in range(c["steps"]):
        f, g = plain.step(f, g, latent, 1.0)
    if c["kind"] == "restart":
        return {"g": g.reshape(7, -1)} if f is None else {"f": f.reshape(19, -1),
                                                         "g": g.reshape(7, -1)}
    h, T, fl, rho, u, _ = plain.macros(f, g, latent)
    out = {"T": T, "fl": fl, "h": h}
    if f is not None:
        out.update(rho=rho, u=u)
    if c["kind"] == "monitor":
        out["scalars"] = {k: None for k in ("liquid_vol", "nu_hot", "front_mean", "sum_h",
                                            "nu_fd", "front_mid")}
        area = c["ny"] * c["nz"]
        out["scalars"].update(liquid_vol=float(fl.sum()), front_mean=float(fl.sum()) / area,
                              sum_h=float(h.sum()),
                              nu_fd=c["nx"] * float((2 * (1 - T[:, :, 0])).sum()) / area)
    return out
