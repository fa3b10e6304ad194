"""The workloads whose speed is measured: what a user's program has this library do.

A case names a flow, a precision form, a grid and the options that are on.  Its
inputs are made here from the seed alone (the recipes follow the workload
descriptions in ``synthetic/workloads.py``; the random part is torch's
generator), `run` passes them through the public entry points, and `exact`
works the same result out in 64-bit torch, from the equations and without the
library.

kind      : steps    K calls of rossbi_step from a stored state, the first
                     with a given step length, the rest with the
                     device-resident CFL step (a time loop's inner part);
                     `monitor` reads the next step length and the
                     conservation sums back, as a loop that logs does.
            host     rossbi_step_host on a state in pinned host memory.
            adjoint  one rossbi_adjoint_step with the derivative in the
                     Stokes number.
            gradient adjoint.run_steps over K steps and its backward pass.
flow      : sod        shock tube in a Box, at a random time of its solution
            explosion  radial shock tube on the polar mesh, one z cell
            disc       stratified Keplerian disc, 1e-4 density noise
            rwi        the disc with a radial density bump and a mode-m seed
            vortex     disc with Gaussian vortices, gas and dust
"""
import math

import numpy as np
import torch

import synthetic as syn
from paper_2207_04252_gb300 import adjoint, rossbi, workloads

PI = math.pi
FORMS = {"f64": rossbi.ROSSBI_FP64, "f32": rossbi.ROSSBI_FP32_PERT, "f64pert": rossbi.ROSSBI_FP64_PERT}
BASE = dict(kind="steps", flow="vortex", form="f64", recon="conservative", nr=0, nth=0, nz=1, dust=0, steps=1,
            gamma=1.4, law=0, monitor=False, indirect=0.0, zones=False, vertical=False)
MU, MV, MW, EN, RHO = range(5)
PERIODIC, OUTFLOW, EQUILIBRIUM = syn.BC_PERIODIC, syn.BC_OUTFLOW, syn.BC_EQUILIBRIUM


def _case(name=None, **kw):
    c = dict(BASE, **kw)
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # the smallest call: the Sod tube of the tests, a launch-bound time loop
        _case("sod_loop_f64", flow="sod", nr=256, nth=4, nz=4, steps=4),
        # a small bi-fluid disc in the fast form (a parameter study's grid): fewer tiles than the GPU has room for
        _case("small_vortex_f32", form="f32", nr=32, nth=48, nz=32, dust=1, steps=4),
        # the stratified gas disc of the tests in the reference form, logged each step
        _case("disc_f64", flow="disc", nr=128, nth=256, nz=32, monitor=True),
        # the Rossby wave instability's gas disc in the fast form, with the reconstruction its long runs use
        _case("rwi_f32_primitive", flow="rwi", form="f32", recon="primitive", nr=256, nth=256, nz=16, steps=2),
        # the bi-fluid vortex of the tests in the fast form
        _case("vortex_f32", form="f32", nr=256, nth=512, nz=64, dust=1, monitor=True),
        # the benchmark's grid: production runs of the fast form
        _case("two_vortices_f32", form="f32", nr=512, nth=1024, nz=128, dust=1),
        # the bi-fluid vortex in the reference form
        _case("vortex_f64", nr=128, nth=256, nz=32, dust=1),
        # the perturbation form in double on a ragged grid
        _case("ragged_vortex_f64pert", form="f64pert", nr=93, nth=131, nz=37, dust=1),
        # the cylindrical explosion at the paper's size: 2-D, shocks, no equilibrium
        _case("explosion_f64", flow="explosion", nr=1600, nth=3200, nz=1),
        # three dust species with the optional terms on, on a ragged grid
        _case("species_f32_options", form="f32", nr=150, nth=211, nz=45, dust=3, law=2, indirect=0.7, zones=True,
              vertical=True),
        # a host program that keeps its state in its own memory
        _case("host_step_f32", kind="host", form="f32", recon="primitive", nr=192, nth=384, nz=48, dust=1),
        # the adjoint workload: a checkpointed gradient through steps of the reference form
        _case("gradient_f64", kind="gradient", nr=128, nth=256, nz=32, dust=1, steps=2),
    ]


def draw(rng):
    """One more case of the same ranges; double-precision and adjoint grids are
    the smaller ones, as their cells cost more, and a disc has the 20 vertical
    cells or more that its Gaussian atmosphere needs to stay physical."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("steps", "steps", "steps", "steps", "steps", "host", "adjoint", "gradient"))
    if kind in ("adjoint", "gradient"):
        return _case(kind=kind, nr=size(28, 100), nth=size(32, 160), nz=size(20, 32), dust=rng.choice((0, 1, 1)),
                     steps=2 if kind == "gradient" else 1, law=rng.choice((0, 1)),
                     recon=rng.choice(("conservative", "primitive")))
    if kind == "host":
        return _case(kind=kind, form=rng.choice(("f32", "f32", "f64")), recon="primitive", nr=size(28, 128),
                     nth=size(32, 256), nz=size(20, 40), dust=rng.choice((0, 1)))
    flow = rng.choice(("sod", "explosion", "disc", "rwi", "vortex", "vortex", "vortex", "vortex"))
    if flow == "sod":
        return _case(flow=flow, form=rng.choice(("f64", "f32")), nr=size(64, 2048), nth=size(1, 12), nz=size(1, 12),
                     steps=rng.choice((1, 2, 4)), gamma=rng.choice((1.4, 1.4, 5.0 / 3.0)))
    if flow == "explosion":
        return _case(flow=flow, nr=size(100, 1600), nth=size(200, 2400), recon=rng.choice(("conservative", "primitive")))
    form = rng.choice(("f32", "f32", "f32", "f64", "f64pert"))
    big = form == "f32"
    c = _case(flow=flow, form=form, nr=size(28, 400 if big else 128), nth=size(32, 800 if big else 256),
              nz=size(20, 100 if big else 36), recon=rng.choice(("conservative", "primitive")),
              steps=rng.choice((1, 1, 2)), monitor=rng.random() < 0.4, gamma=rng.choice((1.4, 1.4, 1.4, 5.0 / 3.0)))
    if flow == "vortex":
        c["dust"] = rng.choice((0, 1, 1, 1, 2, 3))
        c["law"] = rng.choice((0, 0, 1, 2)) if c["dust"] else 0
    if rng.random() < 0.25:
        c.update(indirect=rng.choice((0.0, 0.7)), zones=rng.random() < 0.6, vertical=rng.random() < 0.4)
    return c


def _fields(c):
    return 5 + 4 * c["dust"]


def work(case):
    """Bytes: a step reads E^n and writes E*, then reads both and writes
    E^{n+1} (5 state accesses); the adjoint step reads E^n and a cotangent and
    writes one.  Operations of one cell and stage: 700 for the gas (three
    faces with their reconstruction, one evaluation of the star-pressure
    functions and the flux, and the sources), 270 for each dust species; the
    adjoint of a stage twice those of the stage."""
    cells = case["nr"] * case["nth"] * case["nz"]
    state = _fields(case) * cells * (4 if case["form"] == "f32" else 8)
    flops = 2.0 * cells * (700 + 270 * case["dust"])
    if case["kind"] == "adjoint":
        return {"bytes": 3.0 * state, "flops": 3.0 * flops}
    if case["kind"] == "gradient":
        return {"bytes": (5.0 + 3.0) * state * case["steps"], "flops": 4.0 * flops * case["steps"]}
    return {"bytes": 5.0 * state * case["steps"], "flops": flops * case["steps"]}


# ------------------------------------------------------------------ inputs
DISC = (1.0, -0.5, 0.05 * 0.05 / 2.0, -1.0)
STOKES, KAPPA = 0.1, 0.3
FACTORS = (1.0, 0.3, 3.0, 0.1)
ZONES, VERTICAL = (0.625, 1.68, 1.0), (0.1, 1.0)
SOD_WAVES = (-1.18322, -0.07027, 0.92745, 1.75216)  # head, tail, contact, shock (gamma = 1.4)


class _Setup:
    """Mesh, metric and equilibrium of a case, in 64 bits on `dev` (arrays broadcast over (nz, nth, nr))."""

    def __init__(self, c, dev):
        self.c, self.dev = c, dev
        self.n = (c["nr"], c["nth"], c["nz"])
        self.cyl = c["flow"] != "sod"
        self.disc = c["flow"] in ("disc", "rwi", "vortex")
        self.bump = (0.5, 1.0, 0.025) if c["flow"] == "rwi" else (0.0, 1.0, 0.0)
        self.gamma, self.cfl = c["gamma"], 0.5
        self.gm, self.omega = (1.0 if self.disc else 0.0), 0.0
        if c["flow"] == "sod":
            self.x0, self.x1 = (0.0, 0.0, 0.0), (1.0, self.n[1] / self.n[0], self.n[2] / self.n[0])
        elif c["flow"] == "explosion":
            self.x0, self.x1 = (math.exp(-PI), 0.0, -0.5), (1.0, 2.0 * PI, 0.5)
        else:
            lo, hi, z = (0.6, 1.6, 0.1) if c["flow"] == "rwi" else (0.5, 2.0, 0.15)
            self.x0, self.x1 = (lo, 0.0, -z), (hi, 2.0 * PI, z)
            self.omega = 1.0 if c["flow"] == "vortex" else 2.0 / (lo ** 1.5 + hi ** 1.5)
        edge = EQUILIBRIUM if self.disc else OUTFLOW
        self.bc = (edge, PERIODIC, EQUILIBRIUM if self.disc else PERIODIC)
        nr, nth, nz = self.n
        self.h = [(b - a) / m for a, b, m in zip(self.x0, self.x1, self.n)]
        i = np.arange(-2, nr + 3)
        if self.cyl:
            f = self.x0[0] * (self.x1[0] / self.x0[0]) ** (i / nr)
            cen = np.sqrt(f[:-1] * f[1:])
        else:
            f = self.x0[0] + self.h[0] * i
            cen = 0.5 * (f[:-1] + f[1:])
        self.f_all, self.c_all = f, cen
        rf, self.r = f[2:nr + 3], cen[2:nr + 2]
        self.th = self.x0[1] + (np.arange(nth) + 0.5) * self.h[1]
        self.z = self.x0[2] + (np.arange(nz) + 0.5) * self.h[2]
        if self.cyl:
            base = 0.5 * (rf[1:] ** 2 - rf[:-1] ** 2)
            vol, ar = base * self.h[1] * self.h[2], rf * self.h[1] * self.h[2]
            at, az = (rf[1:] - rf[:-1]) * self.h[2], base * self.h[1]
        else:
            vol, ar = np.full(nr, self.h[0] * self.h[1] * self.h[2]), np.full(nr + 1, self.h[1] * self.h[2])
            at, az = np.full(nr, self.h[0] * self.h[2]), np.full(nr, self.h[0] * self.h[1])
        self.vol, self.area = self.t(vol), [self.t(ar), self.t(at), self.t(az)]
        self.max_area = self.t(np.maximum(ar[1:], np.maximum(at, az)))
        zf = self.x0[2] + np.arange(nz + 1) * self.h[2]
        self.e0 = self.t(self.equilibrium(self.r[None, :], self.z[:, None]))     # (5, nz, nr)
        self.e0r = self.t(self.equilibrium(rf[None, :], self.z[:, None]))
        self.e0z = self.t(self.equilibrium(self.r[None, :], zf[:, None]))

    def t(self, a):
        return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).to(self.dev)

    def primitive(self, r, z):
        """Equilibrium (rho, v_theta in the frame, P) of the disc."""
        s0, bs, t0, bt = DISC
        cs2, om = t0 * r ** bt, np.sqrt(self.gm / r ** 3)
        R = np.sqrt(r * r + z * z)
        pot = 1.0 / R - 1.0 / r
        rho = s0 * r ** bs / (math.sqrt(PI) * np.sqrt(2.0 * cs2) / om) * np.exp(self.gm / cs2 * pot)
        slope = (bt + bs - 0.5 * (bt + 3.0)) / r + self.gm / cs2 * (-bt * pot / r - r / R ** 3 + 1.0 / r ** 2)
        delta, rb, width = self.bump
        if delta:
            x = (r - rb) / width
            G = np.exp(-0.5 * x * x)
            rho = rho * (1.0 + delta * G)
            slope = slope - delta * G * x / (width * (1.0 + delta * G))
        v = np.sqrt(self.gm * r * r / R ** 3 + r * cs2 * slope) - self.omega * r
        return rho, v, cs2 * rho

    def equilibrium(self, r, z):
        out = np.zeros((5,) + np.broadcast_shapes(r.shape, z.shape))
        if self.disc:
            rho, v, p = self.primitive(r, z)
            out[MV], out[EN], out[RHO] = rho * v, 0.5 * rho * v * v + p / (self.gamma - 1.0), rho
        return out


def _smooth(s, gen, modes=4):
    """A sum of random low-order waves of order 1, (nz, nth, nr)."""
    x = s.t((np.log(s.r) - math.log(s.r[0])) / max(1e-9, math.log(s.r[-1] / s.r[0])) if s.cyl else s.r)[None, None, :]
    y, z = s.t(2.0 * PI * np.arange(s.n[1]) / s.n[1])[None, :, None], s.t(np.arange(s.n[2]) / s.n[2])[:, None, None]
    out = torch.zeros(s.n[::-1], dtype=torch.float64, device=s.dev)
    for _ in range(modes):
        k = torch.randint(1, 5, (3,), generator=gen).tolist()
        ph = (2.0 * PI * torch.rand(3, generator=gen, dtype=torch.float64)).tolist()
        out += torch.sin(PI * k[0] * x + ph[0]) * torch.cos(k[1] * y + ph[1]) * torch.cos(PI * k[2] * z + ph[2])
    return out / math.sqrt(modes)


def _inputs(case, seed, dev):
    """(setup, departure E - E0 in 64 bits, CFL step length)."""
    c = dict(BASE, **case)
    s = _Setup(c, dev)
    gen = torch.Generator().manual_seed(seed)
    dgen = torch.Generator(device=dev).manual_seed(seed)
    shape = s.n[::-1]

    def white():
        return 2.0 * torch.rand(shape, generator=dgen, dtype=torch.float64, device=dev) - 1.0

    Ep = torch.zeros((_fields(c),) + shape, dtype=torch.float64, device=dev)
    rho0, v0 = s.e0[RHO][:, None, :], None
    if s.disc:
        v0 = (s.e0[MV] / s.e0[RHO])[:, None, :]
    if c["flow"] in ("sod", "explosion"):  # the tube's waves a random time after the start, 1e-3 noise
        time = 0.04 + 0.08 * torch.rand(1, generator=gen).item()
        xi = (s.r - (0.5 if c["flow"] == "sod" else 0.4)) / time
        head, tail, contact, shock = SOD_WAVES
        u = np.where(xi < tail, np.clip((xi + 1.18322) / 1.2, 0.0, None), np.where(xi < shock, contact, 0.0))
        fan = np.clip(1.0 - 0.2 * u / 1.18322, 0.0, None)
        rho = np.where(xi < tail, fan ** 5, np.where(xi < contact, 0.42632, np.where(xi < shock, 0.26557, 0.125)))
        p = np.where(xi < tail, fan ** 7, np.where(xi < shock, 0.30313, 0.1))
        rho = s.t(rho)[None, None, :] * (1.0 + 1e-3 * white())
        u = s.t(u)[None, None, :] + 1e-3 * _smooth(s, gen)
        v = 1e-3 * _smooth(s, gen)
        Ep[RHO], Ep[MU], Ep[MV] = rho, rho * u, rho * v
        Ep[EN] = s.t(p)[None, None, :] / (s.gamma - 1.0) + 0.5 * rho * (u * u + v * v)
    elif c["flow"] == "disc":
        d = 1e-4 * white() * rho0
        Ep[RHO], Ep[MV], Ep[EN] = d, d * v0, 0.5 * d * v0 * v0
    elif c["flow"] == "rwi":
        r, th = s.t(s.r)[None, None, :], s.t(s.th)[None, :, None]
        ph = 2.0 * PI * torch.rand(1, generator=gen).item()
        G = torch.exp(-0.5 * ((r - 1.0) / 0.025) ** 2)
        u = 1e-4 * (v0 + s.omega * r) * torch.sin(4.0 * th + ph) * G + 1e-7 * _smooth(s, gen)
        Ep[MU], Ep[EN] = rho0 * u, 0.5 * rho0 * u * u
    else:
        r, th = s.t(s.r)[None, None, :], s.t(s.th)[None, :, None]
        up, vp = torch.zeros(1, 1, 1, device=dev), torch.zeros(1, 1, 1, device=dev)
        for rv in (0.8, 1.3) if s.n[0] >= 400 else (1.0,):
            tv = 2.0 * PI * torch.rand(1, generator=gen).item()
            om = rv ** -1.5
            sr = 2.0 * math.sqrt(2.0 * DISC[2] * rv ** DISC[3]) / om
            st = 4.0 * sr
            psi0 = -0.2 * 1.5 * om / (1.0 / sr ** 2 + 1.0 / st ** 2)
            dth = torch.remainder(th - tv + PI, 2.0 * PI) - PI
            psi = psi0 * torch.exp(-(r - rv) ** 2 / (2.0 * sr ** 2) - (rv * dth) ** 2 / (2.0 * st ** 2))
            up, vp = up - psi * rv * rv * dth / (r * st ** 2), vp + psi * (r - rv) / sr ** 2
        d = 1e-4 * rho0 * _smooth(s, gen)  # what a few steps leave of density waves
        if c["kind"] in ("adjoint", "gradient"):  # and a flow without exact limiter ties
            d = d + 1e-4 * rho0 * white()
            up, vp = up + 1e-5 * white(), vp + 1e-5 * white()
            Ep[MW] = (rho0 + d) * (1e-5 * white())
        rho, v = rho0 + d, v0 + vp
        Ep[RHO], Ep[MU] = d, rho * up
        Ep[MV] = d * v0 + rho * vp
        Ep[EN] = 0.5 * rho * (up * up + v * v) - 0.5 * rho0 * v0 * v0 + 0.5 * Ep[MW] ** 2 / rho
        for k in range(c["dust"]):
            b = 5 + 4 * k
            rd = 0.01 / c["dust"] * rho0 * (1.0 + 1e-3 * white())
            Ep[b + 3], Ep[b], Ep[b + 1] = rd, rd * up, rd * v
            if c["kind"] in ("adjoint", "gradient"):
                Ep[b + 2] = rd * (1e-5 * white())
    if c["form"] == "f32":
        Ep = Ep.float().double()
    dt = math.inf
    for a in range(0, s.n[2], 16):  # in slices: the temporaries of the largest grid stay small
        E = Ep[:, a:a + 16].clone()
        E[:5] += s.e0[:, a:a + 16, None, :]
        dt = min(dt, float(_cell_dt(s, E).min()))
    return s, Ep, dt


def _grid(s, form):
    c = s.c
    w = syn.Workload(
        name="case", geometry=syn.GEOM_CYL if s.cyl else syn.GEOM_BOX, nr=s.n[0], nth=s.n[1], nz=s.n[2],
        x0=s.x0, x1=s.x1, bc_lo=s.bc, bc_hi=s.bc, ic="rwi" if c["flow"] == "rwi" else "vortex", steps=c["steps"],
        gamma=s.gamma, gm=s.gm, omega_frame=s.omega, cfl=s.cfl, n_dust=c["dust"], disc=DISC if s.disc else None,
        stokes=STOKES, drag_law=c["law"], drag_kappa=KAPPA, rwi_delta=s.bump[0], rwi_r0=s.bump[1],
        rwi_width=s.bump[2], dust_stokes_factors=FACTORS[:c["dust"]] if c["dust"] > 1 else (),
        recon=syn.RECON_PRIMITIVE if c["recon"] == "primitive" else syn.RECON_CONSERVATIVE)
    g = workloads.Grid(w, precision=FORMS[form])
    if c["indirect"]:
        g.set_indirect(c["indirect"])
    if c["zones"]:
        g.set_damping(ZONES)
    if c["vertical"]:
        g.set_vertical_damping(VERTICAL)
    return g


def _cotangent(s, Ep, seed):
    """A cotangent of order one in each field's own units."""
    E = Ep.clone()
    E[:5] += s.e0[:, :, None, :]
    gen = torch.Generator(device=Ep.device).manual_seed(seed + 77)
    lam = torch.randn(E.shape, generator=gen, dtype=torch.float64, device=E.device)
    return lam / (E.abs().mean(dim=(1, 2, 3), keepdim=True) + 1e-30)


def prepare(case, seed):
    c = dict(BASE, **case)
    s, Ep, dt = _inputs(c, seed, "cuda")
    grid = _grid(s, c["form"])
    if c["form"] == "f64":
        Ep[:5] += s.e0[:, :, None, :]
    E0 = Ep.to(grid.dtype).contiguous()
    st = {"case": c, "grid": grid, "E0": E0, "dt": dt}
    if c["kind"] == "host":
        st["host"] = torch.empty(E0.shape, dtype=E0.dtype, pin_memory=True).copy_(E0).numpy()
        del st["E0"]
    elif c["kind"] in ("adjoint", "gradient"):
        st["lam"] = _cotangent(s, E0 - torch.cat([s.e0, s.e0.new_zeros(E0.shape[0] - 5, *s.e0.shape[1:])])[:, :, None, :],
                               seed)
        if c["kind"] == "adjoint":
            st["out"] = torch.empty_like(E0)
        else:
            st["stokes"] = torch.tensor(STOKES, dtype=torch.float64, requires_grad=True)
            E0.requires_grad_(True)
    else:
        st["E"] = torch.empty_like(E0)
    return st


def run(state):
    c, grid, dt = state["case"], state["grid"], state["dt"]
    if c["kind"] == "host":
        nxt = rossbi.rossbi_step_host(grid.h, state["host"], dt, grid.dust)
        return {"E": state["host"], "dt": nxt}
    if c["kind"] == "adjoint":
        dst = grid.adjoint_step(state["E0"], dt, state["lam"], state["out"], want_dstokes=True)
        return {"lam": state["out"], "dstokes": dst}
    if c["kind"] == "gradient":
        E = adjoint.run_steps(grid, state["E0"], [0.9 * dt] * c["steps"], state["stokes"], every=2)
        lam, dst = torch.autograd.grad((E * state["lam"]).sum(), (state["E0"], state["stokes"]))
        return {"E": E.detach(), "lam": lam, "dstokes": dst}
    E = state["E"]
    E.copy_(state["E0"])
    nxt = None
    for k in range(c["steps"]):
        nxt = grid.step(E, dt=dt if k == 0 else 0.0, want_next_dt=c["monitor"] and k == c["steps"] - 1)
    return {"E": E, "dt": nxt, "sums": grid.sums(E)} if c["monitor"] else {"E": E}


# ------------------------------------------------------------------ the same in 64 bits
def _minmod(a, b):
    return torch.where(a * b <= 0, torch.zeros_like(a), torch.where(a.abs() < b.abs(), a, b))


def _prim(g, U):
    """(u, v, w, P, rho) of a conservative gas state, fields first."""
    ir = 1.0 / U[RHO]
    p = (g - 1.0) * (U[EN] - 0.5 * (U[MU] ** 2 + U[MV] ** 2 + U[MW] ** 2) * ir)
    return torch.stack([U[MU] * ir, U[MV] * ir, U[MW] * ir, p, U[RHO]])


def _cell_dt(s, E):
    W = _prim(s.gamma, E[:5])
    rate = (torch.sqrt(W[0] ** 2 + W[1] ** 2 + W[2] ** 2) + torch.sqrt(s.gamma * W[3] / W[4]))
    for b in range(5, E.shape[0], 4):
        vd = torch.sqrt(E[b] ** 2 + E[b + 1] ** 2 + E[b + 2] ** 2) / E[b + 3].clamp_min(1e-300)
        rate = torch.maximum(rate, vd)
    return s.cfl * s.vol / (rate * s.max_area)


def _pad(q, dim, bc, n=2):
    """`n` ghost cells on both ends of a departure array: periodic, zero gradient, or none (equilibrium)."""
    m = q.shape[dim]
    if bc == PERIODIC:
        at = torch.arange(-n, m + n, device=q.device) % m
    else:
        at = torch.arange(-n, m + n, device=q.device).clamp(0, m - 1)
    out = q.index_select(dim, at)
    if bc == EQUILIBRIUM:
        keep = torch.ones(m + 2 * n, dtype=q.dtype, device=q.device)
        keep[:n] = keep[m + n:] = 0.0
        out = out * keep.view([-1 if d == dim else 1 for d in range(q.dim())])
    return out


def _pressure(g, K, p):
    """f_K(p) and its derivative for side K = (rho, u, p, c)."""
    rar = p <= K[2]
    e = (p / K[2]) ** ((g - 1.0) / (2.0 * g))
    q = torch.sqrt(2.0 / ((g + 1.0) * K[0]) / ((g - 1.0) / (g + 1.0) * K[2] + p))
    f = torch.where(rar, 2.0 * K[3] / (g - 1.0) * (e - 1.0), (p - K[2]) * q)
    d = torch.where(rar, e / (p / K[2] * K[0] * K[3]), (1.0 - 0.5 * (p - K[2]) / ((g - 1.0) / (g + 1.0) * K[2] + p)) * q)
    return f, d


def _riemann(g, L, R):
    """Exact solution at x / t = 0 of the states (rho, u, p); differentiable (implicit function theorem at p*)."""
    L, R = L + (torch.sqrt(g * L[2] / L[0]),), R + (torch.sqrt(g * R[2] / R[0]),)
    with torch.no_grad():
        least = 1e-8 * torch.minimum(L[2], R[2])
        p = 0.5 * (L[2] + R[2]) - 0.125 * (R[1] - L[1]) * (L[0] + R[0]) * (L[3] + R[3])
        p = torch.maximum(p, least)
        for _ in range(60):
            (fl, dl), (fr, dr) = _pressure(g, L, p), _pressure(g, R, p)
            new = torch.maximum(p - (fl + fr + R[1] - L[1]) / (dl + dr), least)
            done = float(((new - p).abs() / (new + p)).max()) < 1e-15
            p = new
            if done:
                break
    (fl, dl), (fr, dr) = _pressure(g, L, p), _pressure(g, R, p)
    p = p - (fl + fr + R[1] - L[1]) / (dl + dr).detach()
    fl, fr = _pressure(g, L, p)[0], _pressure(g, R, p)[0]
    us = 0.5 * (L[1] + R[1]) + 0.5 * (fr - fl)
    g6, out = (g - 1.0) / (g + 1.0), []
    for K, sg in ((L, 1.0), (R, -1.0)):
        x = p / K[2]
        star_r, star_s = K[0] * x ** (1.0 / g), K[0] * (x + g6) / (x * g6 + 1.0)
        cf = (2.0 / (g + 1.0) * (K[3] + sg * 0.5 * (g - 1.0) * K[1])).clamp_min(1e-30)
        fan = (K[0] * (cf / K[3]) ** (2.0 / (g - 1.0)), sg * cf, K[2] * (cf / K[3]) ** (2.0 * g / (g - 1.0)))
        shock = x > 1.0
        speed = torch.where(shock, sg * K[1] - K[3] * torch.sqrt((g + 1.0) / (2.0 * g) * x + (g - 1.0) / (2.0 * g)),
                            sg * K[1] - K[3])
        outside = speed >= 0.0
        inside = ~shock & ~outside & (sg * us - K[3] * x ** ((g - 1.0) / (2.0 * g)) >= 0.0)
        pick = lambda o, f, a: torch.where(outside, o, torch.where(inside, f, a))  # noqa: E731
        out.append((pick(K[0], fan[0], torch.where(shock, star_s, star_r)), pick(K[1], fan[1], us), pick(K[2], fan[2], p)))
    left = us >= 0.0
    return [torch.where(left, a, b) for a, b in zip(*out)], left


def _parabola(q, w, dim):
    """Lower and upper face values of the limited parabola in all cells but the first and last."""
    m = q.shape[dim]
    qm, q0, qp = (q.narrow(dim, a, m - 2) for a in range(3))
    sm, sp = (q0 - qm) * w[0], (qp - q0) * w[1]
    s, a, b = _minmod(sm, sp), (sp - sm) * w[2], (sp * w[3] + sm * w[4]) * w[2]
    return q0 + _minmod(w[5] * (a * w[5] + b), s * w[7]), q0 + _minmod(w[6] * (a * w[6] + b), s * w[8])


def _divergence(s, E, axis, j0, j1):
    """Sum of A F over the lower minus the upper face along `axis` of the cells j0 .. j1 - 1 of axis 1."""
    c, g, dim = s.c, s.gamma, 3 - axis
    prim = c["recon"] == "primitive"
    n = s.n[axis]
    if axis == 1:
        rows = torch.arange(j0 - 2, j1 + 2, device=E.device) % s.n[1]
        E, n = E.index_select(2, rows), j1 - j0
    else:
        E = E[:, :, j0:j1]
    e0 = s.e0[:, :, None, :]
    gas = _prim(g, E[:5]) - (_prim(g, e0) if s.disc else 0.0) if prim else E[:5] - e0
    dust = []
    for b in range(5, E.shape[0], 4):
        rd = E[b + 3]
        ir = torch.where(rd > 0, 1.0 / torch.where(rd > 0, rd, torch.ones_like(rd)), torch.zeros_like(rd))
        dust.append(torch.stack([E[b] * ir, E[b + 1] * ir, E[b + 2] * ir, rd]))
    q = torch.cat([gas] + dust)
    if axis != 1:
        q = _pad(q, dim, s.bc[axis])
    if axis == 0:
        x, f = s.c_all, s.f_all
        xm, x0, xp, fm, fp = x[:-2], x[1:-1], x[2:], f[1:-2], f[2:-1]
        w = [s.t(v) for v in (1 / (x0 - xm), 1 / (xp - x0), 1 / (xp - xm), x0 - xm, xp - x0, fm - x0, fp - x0,
                              -np.minimum(2 * (x0 - fm), x0 - xm), np.minimum(2 * (fp - x0), xp - x0))]
    else:
        h = s.h[axis]
        w = [1 / h, 1 / h, 0.5 / h, h, h, -0.5 * h, 0.5 * h, -h, h]
    lo, hi = _parabola(q, w, dim)                     # cells -1 .. n
    mid = q.narrow(dim, 1, n + 2)
    if axis == 0:
        f0, area = s.e0r[:, :, None, :], s.area[0]
    elif axis == 1:
        f0, area = s.e0[:, :, None, :], s.area[1]
    else:
        f0, area = s.e0z[:, :, None, :], s.area[2]
    if prim and s.disc:
        f0 = _prim(g, f0)

    def at(first):  # the face equilibrium of the cells' lower (first = -1) or upper (0) faces
        if axis == 1:
            return f0
        return f0.index_select(dim, torch.arange(first, first + n + 2, device=E.device).clamp(0, n))

    def states(l, h):
        a, b = at(-1) + l[:5], at(0) + h[:5]
        return (a, b) if prim else (_prim(g, a), _prim(g, b))

    a, b = states(lo, hi)
    ok = (a[RHO] > 0) & (b[RHO] > 0) & (a[EN] > 0) & (b[EN] > 0)
    if not bool(ok.all()):
        fa, fb = states(mid, mid)
        a, b = torch.where(ok, a, fa), torch.where(ok, b, fb)
    WL, WR = b.narrow(dim, 0, n + 1), a.narrow(dim, 1, n + 1)
    t = [k for k in (MU, MV, MW) if k != axis]
    (rho, u, p), left = _riemann(g, (WL[RHO], WL[axis], WL[EN]), (WR[RHO], WR[axis], WR[EN]))
    t1, t2 = (torch.where(left, WL[k], WR[k]) for k in t)
    F = [None] * 5
    F[RHO], F[axis], F[t[0]], F[t[1]] = rho * u, rho * u * u + p, rho * u * t1, rho * u * t2
    F[EN] = (0.5 * rho * (u * u + t1 * t1 + t2 * t2) + g / (g - 1.0) * p) * u
    for k in range(5, E.shape[0], 4):
        DL, DR = hi[k:k + 4].narrow(dim, 0, n + 1), lo[k:k + 4].narrow(dim, 1, n + 1)
        ml, mr = DL[3] * DL[axis].clamp_min(0.0), DR[3] * DR[axis].clamp_max(0.0)
        F += [ml * DL[q] + mr * DR[q] for q in range(3)] + [ml + mr]
    F = torch.stack(F) * area
    return F.narrow(dim, 0, n) - F.narrow(dim, 1, n)


def _sources(s, E, grad):
    """Geometric, gravity and frame sources per unit volume; grad: the indirect potential's gradient or None."""
    r, z = s.t(s.r)[None, None, :], s.t(s.z)[:, None, None]
    R3 = (r * r + z * z) ** 1.5
    fr, fz, om = -s.gm * r / R3, -s.gm * z / R3, s.omega
    W = _prim(s.gamma, E[:5])
    out = []
    for b in [0] + list(range(5, E.shape[0], 4)):
        rho = E[RHO] if b == 0 else E[b + 3]
        ir = torch.where(rho > 0, 1.0 / torch.where(rho > 0, rho, torch.ones_like(rho)), torch.zeros_like(rho))
        u, v, w = E[b] * ir, E[b + 1] * ir, E[b + 2] * ir
        S = [rho * (v * v / r + fr + 2.0 * om * v + om * om * r), -rho * u * (v / r + 2.0 * om), rho * fz]
        if b == 0:
            S[0] = S[0] + W[EN] / r
            S += [rho * u * (fr + om * om * r) + rho * w * fz, torch.zeros_like(rho)]
        else:
            S += [torch.zeros_like(rho)]
        if grad is not None:
            S[0], S[1] = S[0] - rho * grad[0], S[1] - rho * grad[1]
            if b == 0:
                S[3] = S[3] - rho * (u * grad[0] + v * grad[1])
        out += S
    return torch.stack(out)


def _rhs(s, E, grad, slab, whole=True):
    """G(E) (sum of face fluxes plus V S), in slabs of axis 1."""
    parts = []
    for j0 in range(0, E.shape[2] if whole else 1, slab):
        j1 = min(E.shape[2], j0 + slab) if whole else 1
        G = sum(_divergence(s, E, axis, j0, j1) for axis in range(3))
        if s.cyl:
            G = G + s.vol * _sources(s, E[:, :, j0:j1], None if grad is None else [v[:, j0:j1] for v in grad])
        parts.append(G)
    return parts[0] if len(parts) == 1 else torch.cat(parts, dim=2)


def _drag(s, E, tau, stokes):
    """Backward-Euler drag of the gas and every dust species over tau."""
    nd = (E.shape[0] - 5) // 4
    if not nd:
        return E
    rg, P = E[RHO], _prim(s.gamma, E[:5])[EN]
    if s.c["law"]:
        rho1, _, p1 = s.primitive(np.float64(1.0), np.float64(0.0))
        ts0 = float(rho1 * np.sqrt(s.gamma * p1 / rho1)) / (rg * torch.sqrt(s.gamma * P / rg))
        if s.c["law"] == 2:
            ts0 = torch.where(KAPPA * rg > 2.25, ts0 * (4.0 / 9.0) * KAPPA * rg, ts0)
    else:
        ts0 = s.t(np.sqrt(s.r ** 3 / s.gm))[None, None, :]
    w, den, num = [], rg, [E[k] for k in range(3)]
    for k in range(nd):
        b, a = 5 + 4 * k, tau / (ts0 * stokes * FACTORS[k])
        w.append(a / (1.0 + a))
        den = den + E[b + 3] * w[k]
        num = [num[q] + E[b + q] * w[k] for q in range(3)]
    vg = [m / den for m in num]
    out = [rg * v for v in vg]
    out.append(E[EN] + 0.5 * rg * sum(v * v - (E[q] / rg) ** 2 for q, v in enumerate(vg)))
    out.append(rg)
    for k in range(nd):
        b = 5 + 4 * k
        out += [E[b + q] + E[b + 3] * w[k] * (vg[q] - E[b + q] / E[b + 3]) for q in range(3)] + [E[b + 3]]
    return torch.stack(out)


def _moments_gradient(s, E):
    r, z, th = s.t(s.r)[None, None, :], s.t(s.z)[:, None, None], s.t(s.th)[None, :, None]
    m = E[RHO] - s.e0[RHO][:, None, :]
    for b in range(5, E.shape[0], 4):
        m = m + E[b + 3]
    m = m * (s.vol * r / (r * r + z * z) ** 1.5)
    A, B, X = (m * torch.cos(th)).sum(), (m * torch.sin(th)).sum(), s.c["indirect"]
    return [X * (A * torch.cos(th) + B * torch.sin(th)), X * (-A * torch.sin(th) + B * torch.cos(th))]


def _damping(s):
    if not (s.c["zones"] or s.c["vertical"]):
        return None
    k = np.zeros((s.n[2], s.n[0]))
    lo, hi = s.x0[0], s.x1[0]
    if s.c["zones"]:
        a, b, f = ZONES
        k += np.where(s.r < a, ((a - s.r) / (a - lo)) ** 2 / (2.0 * PI * f * lo ** 1.5), 0.0)
        k += np.where(s.r > b, ((s.r - b) / (hi - b)) ** 2 / (2.0 * PI * f * hi ** 1.5), 0.0)
    if s.c["vertical"]:
        e, f = VERTICAL
        x = np.clip((np.abs(s.z) - e) / (s.x1[2] - e), 0.0, None)[:, None]
        k += x * x / (2.0 * PI * f * s.r ** 1.5)
    return s.t(k)[:, None, :]


def _step(s, E, dt, stokes, R0, damp, slab):
    base, cur = E, E
    for tau in (0.5 * dt, dt):
        grad = _moments_gradient(s, cur) if s.c["indirect"] else None
        G = _rhs(s, cur, grad, slab)
        G = torch.cat([G[:5] - R0, G[5:]])
        if damp is not None:
            G = torch.cat([G[:5] - s.vol * damp * (cur[:5] - s.e0[:, :, None, :]), G[5:]])
        cur = _drag(s, base + tau * G / s.vol, tau, stokes)
    return cur


def exact(case, seed):
    c = dict(BASE, **case)
    cells = c["nr"] * c["nth"] * c["nz"]
    if cells > 20_000_000:  # over the time that a check should take
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    s, Ep, dt = _inputs(c, seed, dev)
    zero = torch.cat([s.e0, s.e0.new_zeros(_fields(c) - 5, *s.e0.shape[1:])])[:, :, None, :]
    E0 = zero + Ep
    R0 = 0.0
    damp = _damping(s)
    slab = max(8, 2_000_000 // (c["nr"] * c["nz"])) if c["kind"] not in ("adjoint", "gradient") else c["nth"]
    if s.disc:
        ring = zero.expand(-1, -1, s.n[1], -1)
        R0 = _rhs(s, ring, None, 1, whole=False)[:5]
    if c["kind"] in ("adjoint", "gradient"):
        lam = _cotangent(s, Ep, seed)
        stokes = torch.tensor(STOKES, dtype=torch.float64, device=dev, requires_grad=True)
        h, K = (dt, 1) if c["kind"] == "adjoint" else (0.9 * dt, c["steps"])
        states = [E0]
        for _ in range(K):
            with torch.no_grad():
                states.append(_step(s, states[-1], h, stokes, R0, damp, slab))
        dst = 0.0
        for k in reversed(range(K)):
            X = states[k].clone().requires_grad_(True)
            ask = (X, stokes) if c["dust"] else (X,)
            got = torch.autograd.grad((_step(s, X, h, stokes, R0, damp, slab) * lam).sum(), ask)
            lam, dst = got[0], dst + (float(got[1]) if c["dust"] else 0.0)
        if c["kind"] == "adjoint":
            return {"lam": lam, "dstokes": dst}
        return {"E": states[-1], "lam": lam, "dstokes": torch.tensor(dst, dtype=torch.float64)}
    E = E0
    for k in range(c["steps"]):
        E = _step(s, E, dt, STOKES, R0, damp, slab)
        dt = float(_cell_dt(s, E).min())
    out = {"E": E if c["form"] == "f64" else E - zero}
    if c["kind"] == "host":
        out["dt"] = dt
    if c["monitor"]:
        out["dt"], out["sums"] = dt, (E * s.vol).sum(dim=(1, 2, 3))
    return out
