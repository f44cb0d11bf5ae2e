"""Workloads whose time is measured: what a program that uses this library has it do.

Three kinds of calls, each through the public binding (`paper_2109_10277_gb300.hq`):

  solve  `Grid.poisson_solve`: Dirichlet Poisson problems on one transverse slice;
  sweep  `Grid.sweep`: a whole quasi-static sweep of a box (a few to some hundred slices), with
         or without field output, witness sums and a beam push;
  grad   `SweepLoss`: a checkpointed sweep and its reverse (autograd), the gradient of a
         witness loss with respect to beam weights, density scale and radial profile.

Boxes keep the cell sizes, slice spacings, shape orders, particles per cell and beams of the
library's named workloads (`inputs.grid_params`); a sweep's work per slice does not depend on
the number of slices, so the boxes are shorter along zeta and their beams sit inside them.
`exact` evaluates the same equations in plain torch and 64 bits.
"""
import math

import torch

from paper_2109_10277_gb300 import hq

AB5 = (1901 / 720, -2774 / 720, 2616 / 720, -1274 / 720, 251 / 720)
MIX, GUARD = 0.05, 0.02     # predictor-corrector mixing and removal threshold of every named workload
GAMMA = 1e10 / 0.51099895e6  # 10 GeV beams


def _solve(name, precision, nx, ny, nrhs):
    return dict(name=name, kind="solve", precision=precision, nx=nx, ny=ny, nrhs=nrhs)


def _sweep(name, precision, nx, ny, nz, **over):
    c = dict(name=name, kind="sweep", precision=precision, nx=nx, ny=ny, nz=nz, half=8.0, dz=0.02, order=2,
             ppc_x=1, ppc_y=1, solver="pc", iters=5, density=5.0, sigma_r=0.2, n_beam=50_000, n_witness=0,
             dt=0.0, ions=False, fields="ez,psi")
    c.update(over)
    return c


def _grad(name, precision, nx, ny, nz, **over):
    c = dict(name=name, kind="grad", precision=precision, nx=nx, ny=ny, nz=nz, half=6.0, dz=0.0234, order=1,
             ppc_x=1, ppc_y=1, iters=5, density=2.0, sigma_r=0.2, n_beam=40_000, n_witness=10_000, ckpt=16,
             loss="mean", profile=0)
    c.update(over)
    return c


def listed():
    return [
        # one small Poisson problem: nothing but launches and latency
        _solve("solve_64", "fp32", 64, 64, 1),
        # psi, Ez and Bz of one slice of the 512^2 workload
        _solve("solve_512", "fp32", 512, 512, 3),
        # a grid that no tile divides, in the more accurate operand split
        _solve("solve_ragged_tf32x3", "tf32x3", 328, 200, 2),
        # a large transverse grid
        _solve("solve_2048", "fp32", 2048, 2048, 2),
        # the double-precision solver at the same slice as the FP32 one
        _solve("solve_fp64_512", "fp64", 512, 512, 2),
        # the linear-regime reference run in double precision, whole
        _sweep("sweep_linear64_fp64", "fp64", 64, 64, 64, half=6.0, dz=0.1875, order=1, density=0.01, sigma_r=0.3,
               n_beam=100_000, n_witness=20_000, fields="ez,psi,bx,by,jz"),
        # the blowout workload in double precision, the arm that FP32 is held against
        _sweep("sweep_blowout512_fp64", "fp64", 512, 512, 12, dz=0.0195, n_witness=10_000),
        # the blowout workload: the call that a production run consists of
        _sweep("sweep_blowout512", "fp32", 512, 512, 96, dz=0.0195, n_beam=200_000, n_witness=20_000, fields="ez"),
        # fine grid, cubic shape, 4 particles per cell, driver and witness pushed: one beam time step
        _sweep("sweep_cubic1024", "fp32", 1024, 1024, 16, half=10.0, dz=0.0234, order=3, ppc_x=2, ppc_y=2,
               density=10.0, sigma_r=0.15, n_beam=1_000_000, n_witness=200_000, dt=20.0, fields=""),
        # one time step of a beam-quality study on a small grid: many short launches
        _sweep("sweep_study128", "fp32", 128, 128, 64, half=6.0, dz=0.0469, order=1, density=0.5, sigma_r=0.4,
               n_beam=200_000, n_witness=50_000, dt=20.0, fields=""),
        # the explicit B_perp solver
        _sweep("sweep_explicit256", "fp32", 256, 256, 32, dz=0.0195, solver="explicit", iters=6, fields="ez,bx,by"),
        # gradient of a witness loss with respect to the beams and the plasma density
        _grad("grad_256", "fp32", 256, 256, 48),
    ]


# ------------------------------------------------------------------------------------- drawn cases
def _cost(c):
    """Rough time of a pass in arbitrary units, only to keep drawn cases under the largest listed one."""
    n2, slow = c["nx"] * c["ny"], 12.0 if c["precision"] == "fp64" else 1.5 if c["precision"] == "tf32x3" else 1.0
    pow2 = all(c[k] & (c[k] - 1) == 0 for k in ("nx", "ny"))
    if c["precision"] == "fp64" and not pow2:
        slow *= max(c["nx"], c["ny"]) / 64.0
    if c["kind"] == "solve":
        return slow * c["nrhs"] * (30000 + n2)
    per = n2 * c["ppc_x"] * c["ppc_y"] * (c["order"] + 1) ** 2 / 9.0 * (2 if c.get("ions") else 1)
    return slow * c["nz"] * (300000 + 6 * (per + n2)) * (5 if c["kind"] == "grad" else 1)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _extent(rng, lo, hi):
    """A grid extent: a power of two, a multiple of 128, or any size."""
    n = _log(rng, lo, hi)
    kind = rng.random()
    if kind < 0.4:
        return 1 << max(5, min(11, round(math.log2(n))))
    if kind < 0.6 and n >= 128:
        return (n + 64) // 128 * 128
    return n


def draw(rng):
    top = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(("solve", "solve", "sweep", "sweep", "sweep", "grad"))
        precision = rng.choice(("fp32", "fp32", "tf32x3", "fp64"))
        if kind == "solve":
            hi = 1024 if precision == "fp64" else 2048
            c = _solve("", precision, _extent(rng, 32, hi), _extent(rng, 32, hi), rng.randint(1, 5))
            if rng.random() < 0.5:
                c["ny"] = c["nx"]
        else:
            nx = _extent(rng, 48, 512 if kind == "sweep" else 256)
            ny = nx if rng.random() < 0.7 else _extent(rng, 48, 512 if kind == "sweep" else 256)
            order = rng.randint(1, 3)
            half = rng.uniform(5.0, 10.0)
            ppc = rng.choice(((1, 1), (1, 1), (2, 1), (2, 2)))
            over = dict(half=half, dz=rng.uniform(0.015, 0.05), order=order, ppc_x=ppc[0], ppc_y=ppc[1],
                        density=rng.uniform(0.05, 5.0), sigma_r=rng.uniform(0.25, 0.5), n_beam=_log(rng, 5000, 200_000))
            if kind == "sweep":
                over["solver"] = rng.choice(("pc", "pc", "pc", "explicit"))
                over["ions"] = rng.random() < 0.2
                over["dt"] = rng.choice((0.0, 0.0, 6.0, 20.0))
                over["n_witness"] = rng.choice((0, _log(rng, 2000, 50_000)))
                over["fields"] = rng.choice(("ez", "ez,psi,bx,by", "rho,jx,jy,jz,chi,psi,exmby,eypbx,ez,bx,by,bz"))
                c = _sweep("", precision, nx, ny, _log(rng, 8, 64), **over)
            else:
                over["loss"] = rng.choice(("mean", "mean+rms"))
                over["profile"] = rng.choice((0, 64))
                over["n_witness"] = _log(rng, 2000, 20_000)
                c = _grad("", precision, nx, ny, _log(rng, 8, 32), ckpt=rng.choice((4, 8, 16)), **over)
        del c["name"]
        if _cost(c) <= top:
            return c


# ------------------------------------------------------------------------------------------ inputs
def _params(c):
    h = c["half"] if "half" in c else 8.0
    p = dict(nx=c["nx"], ny=c["ny"], nzeta=c.get("nz", 1), xmin=-h, xmax=h, ymin=-h, ymax=h, pc_mix=MIX, psi_guard=GUARD)
    length = c.get("nz", 1) * c.get("dz", 1.0)
    p.update(zeta_min=-0.5 * length, zeta_max=0.5 * length)
    if c["kind"] != "solve":
        p.update(shape_order=c["order"], ppc_x=c["ppc_x"], ppc_y=c["ppc_y"], n_pc_iter=c["iters"])
        p["bperp_solver"] = c.get("solver", "pc")
    if c.get("ions"):   # electrons and mobile hydrogen ions placed alike
        p["species"] = [dict(charge=-1.0, mass=1.0, ppc_x=c["ppc_x"], ppc_y=c["ppc_y"], neutralize=False),
                        dict(charge=1.0, mass=1836.15, ppc_x=c["ppc_x"], ppc_y=c["ppc_y"], neutralize=False)]
    if c.get("profile"):
        p.update(radial_profile=[1.0 + 0.1 * math.cos(0.1 * k) for k in range(c["profile"])], profile_rmax=math.sqrt(2.0) * h)
    return p


def _beam(gen, n, sigma_r, sigma_z, zeta0, density, offset, spread):
    r = torch.randn((6, n), generator=gen, dtype=torch.float64, device="cuda")
    g = GAMMA * (1.0 + 1e-3 * r[5])
    w = density * (2.0 * math.pi) ** 1.5 * sigma_r * sigma_r * sigma_z / n
    return dict(x=offset + sigma_r * r[0], y=sigma_r * r[1], zeta=zeta0 + sigma_z * r[2], ux=spread * r[3], uy=spread * r[4],
                uz=torch.sqrt(g * g - 1.0), w=torch.full((n,), w, dtype=torch.float64, device="cuda"))


def _beams(c, seed):
    """Driver in the front half of the box, witness near its tail."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    length = c["nz"] * c["dz"]
    spread = 0.05 if c.get("dt") else 0.0
    b = [_beam(gen, c["n_beam"], c["sigma_r"], length / 7.0, 0.1 * length, c["density"], 0.0, spread)]
    if c["n_witness"]:
        b.append(_beam(gen, c["n_witness"], 0.5 * c["sigma_r"], length / 25.0, -0.3 * length, 2.0 * c["density"],
                       0.25 * c["sigma_r"], spread))
    return b


def _sources(c, seed):
    """Charge-like sources: an off-centre bunch, a channel wall around it, and shot noise."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dt = torch.float64
    x = torch.linspace(-8.0, 8.0, c["nx"] + 1, dtype=dt, device="cuda")[:-1]
    y = torch.linspace(-8.0, 8.0, c["ny"] + 1, dtype=dt, device="cuda")[:-1]
    src = torch.empty((c["nrhs"], c["ny"], c["nx"]), dtype=dt, device="cuda")
    for r in range(c["nrhs"]):
        a = torch.rand(4, generator=gen, dtype=dt, device="cuda")
        r2 = (x[None, :] - 2.0 * a[0] + 1.0) ** 2 + (y[:, None] - 2.0 * a[1] + 1.0) ** 2
        src[r] = 4.0 * torch.exp(-r2 / (0.2 + a[2])) - torch.exp(-(torch.sqrt(r2) - 2.0 - a[3]) ** 2 / 0.1)
    src += 0.02 * torch.randn(src.shape, generator=gen, dtype=dt, device="cuda")
    return src if c["precision"] == "fp64" else src.float()


def prepare(case, seed):
    grid = hq.Grid(_params(case), precision=case["precision"])
    s = dict(case=case, grid=grid)
    if case["kind"] == "solve":
        s["src"] = _sources(case, seed)
        return s
    arrays = _beams(case, seed)
    s["beams"] = [hq.Beam(a) for a in arrays]
    if case["kind"] == "sweep":
        s["start"] = arrays if case["dt"] else None
        if case["dt"]:
            s["beams"] = [hq.Beam({k: v.clone() for k, v in a.items()}) for a in arrays]
        s["out"] = grid.alloc_out(case["fields"].split(",")) if case["fields"] else None
        s["sums"] = torch.zeros(3, dtype=torch.float64, device="cuda")
    else:
        # the parameters of an optimisation, in the grid's own precision
        s["n0"] = torch.ones((), dtype=grid.dtype, device="cuda", requires_grad=True)
        prof = grid.params.get("radial_profile", [])
        s["profile"] = torch.tensor(prof, dtype=grid.dtype, device="cuda", requires_grad=bool(prof))
        s["w"] = [a["w"].to(grid.dtype).requires_grad_() for a in arrays]
    return s


def run(state):
    c, grid = state["case"], state["grid"]
    if c["kind"] == "solve":
        return grid.poisson_solve(state["src"])
    beams = state["beams"]
    if c["kind"] == "grad":
        loss = hq.SweepLoss.apply(grid, beams, 1, c["loss"], c["ckpt"], state["n0"], state["profile"], *state["w"])
        wanted = [state["n0"], *state["w"]] + ([state["profile"]] if c["profile"] else [])
        grads = torch.autograd.grad(loss, wanted)
        return dict(loss=loss.detach().to(grid.dtype), n0=grads[0], w=list(grads[1:1 + len(beams)]), profile=list(grads[1 + len(beams):]))
    if c["dt"]:
        # a time step from the beams in hand: the push works in place
        for b, a in zip(beams, state["start"]):
            for k in ("x", "y", "zeta", "ux", "uy", "uz"):
                b.t[k].copy_(a[k])
    wit = 1 if c["n_witness"] else -1
    if wit >= 0:
        state["sums"].zero_()
    grid.sweep(beams, dt=c["dt"], out=state["out"], witness=wit, witness_sums=state["sums"] if wit >= 0 else None)
    res = dict(state["out"] or {})
    if wit >= 0:
        res["sums"] = state["sums"].to(grid.dtype)   # as exact as the grid's fields
    if c["dt"]:
        res["beams"] = [{k: b.t[k] for k in ("x", "y", "zeta", "ux", "uy", "uz")} for b in beams]
    return res


# --------------------------------------------------------------------------------- necessary work
def work(case):
    """Bytes and operations that the equations need: fields and particles read and written once
    per step of the slice loop, transforms by the fast algorithm (5 N log2 N)."""
    c = case
    t = 8 if c["precision"] == "fp64" else 4
    nn = c["nx"] * c["ny"]
    fft = 4 * 2.5 * nn * (math.log2(c["nx"]) + math.log2(c["ny"])) / 2
    if c["kind"] == "solve":
        return dict(bytes=2.0 * t * nn * c["nrhs"], flops=fft * c["nrhs"])
    npart = nn * c["ppc_x"] * c["ppc_y"] * (2 if c.get("ions") else 1)
    st = (c["order"] + 1) ** 2
    passes = c["iters"] if c.get("solver", "pc") == "pc" else 1
    # plasma state (x, y, Psi in 64 bits, u and the AB5 history) in and out once a slice, and its
    # fields once a pass
    per_particle = 2 * (24 + 2 * t + 20 * t) + (passes + 1) * 6 * t
    part_flops = (passes + 1) * (st * (6 * 2 + 4 * 2) + 80)
    solves = 3 + 2 * c["iters"]
    per_slice_bytes = npart * per_particle + nn * t * (5 + 6 + 4 * solves)
    per_slice_flops = npart * part_flops + solves * fft
    n_out = len(c["fields"].split(",")) if c.get("fields") else 0
    beam = (c["n_beam"] + c["n_witness"]) * 8 * (13 if c.get("dt") else 7)
    times = 4 if c["kind"] == "grad" else 1   # forward, recompute and the transposed steps (twice the forward's)
    return dict(bytes=float(c["nz"] * (times * per_slice_bytes + n_out * nn * t) + beam), flops=float(c["nz"] * times * per_slice_flops))


# ------------------------------------------------------------- the equations in 64 bits, plain torch
class _Ref:
    """The slice loop in FP64: DST-I by its matrix, index_add deposits, one tensor per quantity."""

    def __init__(self, c, n0=None, profile=None):
        self.c, p = c, _params(c)
        self.nx, self.ny, self.nz = c["nx"], c["ny"], c.get("nz", 1)
        self.x0, self.y0, self.x1, self.y1 = p["xmin"], p["ymin"], p["xmax"], p["ymax"]
        self.dx, self.dy = (self.x1 - self.x0) / self.nx, (self.y1 - self.y0) / self.ny
        self.zmax = p["zeta_max"]
        self.dz = (p["zeta_max"] - p["zeta_min"]) / self.nz
        self.kw = dict(dtype=torch.float64, device="cuda")
        self.sx, self.sy = self._sine(self.nx), self._sine(self.ny)
        ex = -4.0 / self.dx ** 2 * torch.sin(math.pi * torch.arange(self.nx, **self.kw) / (2 * self.nx)) ** 2
        ey = -4.0 / self.dy ** 2 * torch.sin(math.pi * torch.arange(self.ny, **self.kw) / (2 * self.ny)) ** 2
        self.lam = ey[:, None] + ex[None, :]
        self.mask = torch.ones((self.ny, self.nx), **self.kw)
        self.mask[0] = 0.0
        self.mask[:, 0] = 0.0
        self.n0, self.profile = n0, profile
        self.area = self.dx * self.dy

    def _sine(self, n):
        j = torch.arange(n, device="cuda", dtype=torch.int64)
        return torch.sin(math.pi * ((j[:, None] * j[None, :]) % (2 * n)).double() / n)

    def solve(self, s, shift=0.0):
        f = self.sy @ (s * self.mask) @ self.sx
        inv = torch.zeros_like(self.lam)
        inv[1:, 1:] = 4.0 / (self.nx * self.ny) / (self.lam[1:, 1:] - shift)
        return self.sy @ (f * inv) @ self.sx

    def ddx(self, f):
        p = torch.nn.functional.pad(f, (1, 1))
        return (p[:, 2:] - p[:, :-2]) / (2 * self.dx) * self.mask

    def ddy(self, f):
        p = torch.nn.functional.pad(f, (0, 0, 1, 1))
        return (p[2:] - p[:-2]) / (2 * self.dy) * self.mask

    # B-splines
    def _w(self, u):
        o = self.c["order"]
        if o in (0, 2):
            j = torch.floor(u.detach() + 0.5)
            d = u - j
            return j.long() - o // 2, [torch.ones_like(u)] if o == 0 else [0.5 * (0.5 - d) ** 2, 0.75 - d * d, 0.5 * (0.5 + d) ** 2]
        j = torch.floor(u.detach())
        d = u - j
        if o == 1:
            return j.long(), [1.0 - d, d]
        return j.long() - 1, [(1 - d) ** 3 / 6, (4 - 6 * d * d + 3 * d ** 3) / 6, (1 + 3 * d + 3 * d * d - 3 * d ** 3) / 6, d ** 3 / 6]

    def _nodes(self, x, y):
        jx, wx = self._w((x - self.x0) / self.dx)
        jy, wy = self._w((y - self.y0) / self.dy)
        for b, wb in enumerate(wy):
            iy = jy + b
            for a, wa in enumerate(wx):
                ix = jx + a
                ok = (ix >= 1) & (ix < self.nx) & (iy >= 1) & (iy < self.ny)
                yield torch.where(ok, iy * self.nx + ix, 0), torch.where(ok, wa * wb, 0.0)

    def deposit(self, x, y, vals):
        out = [torch.zeros(self.ny * self.nx, **self.kw) for _ in vals]
        for i, w in self._nodes(x, y):
            out = [o.index_add(0, i, w * v) if v.requires_grad or w.requires_grad else o.index_add_(0, i, w * v) for o, v in zip(out, vals)]
        return [o.reshape(self.ny, self.nx) for o in out]

    def gather(self, x, y, fields):
        flat = [f.reshape(-1) for f in fields]
        out = [0.0] * len(flat)
        for i, w in self._nodes(x, y):
            out = [o + w * f[i] for o, f in zip(out, flat)]
        return out

    # plasma
    def plasma(self):
        c, kw = self.c, self.kw
        px, py = c["ppc_x"], c["ppc_y"]
        g = torch.meshgrid(torch.arange(self.ny, **kw), torch.arange(self.nx, **kw), torch.arange(py, **kw), torch.arange(px, **kw), indexing="ij")
        x = (self.x0 + (g[1] + (g[3] + 0.5) / px) * self.dx).reshape(-1)
        y = (self.y0 + (g[0] + (g[2] + 0.5) / py) * self.dy).reshape(-1)
        dens = torch.ones_like(x)
        if self.profile is not None:
            n, rmax = self.profile.numel(), _params(c)["profile_rmax"]
            t = torch.clamp(torch.sqrt(x * x + y * y) / rmax * (n - 1), 0.0, float(n - 1))
            k = torch.clamp(torch.floor(t).long(), 0, n - 2)
            dens = self.profile[k] * (1 - (t - k)) + self.profile[k + 1] * (t - k)
        w = dens * (self.area / (px * py))
        if self.n0 is not None:
            w = w * self.n0
        sp = [(-1.0, 1.0)] + ([(1.0, 1836.15)] if c.get("ions") else [])
        z = torch.zeros(x.numel() * len(sp), **kw)
        one = torch.ones_like(x)
        return dict(x=x.repeat(len(sp)), y=y.repeat(len(sp)), ux=z, uy=z, psi=z, w=w.repeat(len(sp)), ok=torch.ones_like(z, dtype=torch.bool),
                    q=torch.cat([q * one for q, _ in sp]), qm=torch.cat([q / m * one for q, m in sp]))

    def rates(self, s, F):
        e, h, ez, bx, by, bz = F
        opp = 1.0 + s["psi"]
        g = 1.0 / opp
        gam = (1.0 + s["ux"] ** 2 + s["uy"] ** 2 + opp * opp) * 0.5 * g
        k = -s["qm"]
        return (-s["ux"] * g, -s["uy"] * g, k * (gam * g * e + by + bz * g * s["uy"]), k * (gam * g * h - bx - bz * g * s["ux"]),
                k * (g * (s["ux"] * e + s["uy"] * h) - ez))

    def step(self, s, f, hist):
        comb = [sum(AB5[k] * h[i] for k, h in enumerate([f] + hist)) for i in range(5)]
        new = [s[k] - self.dz * v for k, v in zip(("x", "y", "ux", "uy", "psi"), comb)]
        x, y, _, _, psi = [t.detach() for t in new]
        ok = s["ok"] & (x > self.x0) & (x < self.x1) & (y > self.y0) & (y < self.y1) & (1.0 + psi >= GUARD)
        new = [torch.where(ok, t, s[k]) for k, t in zip(("x", "y", "ux", "uy", "psi"), new)]
        return dict(s, ok=ok, **dict(zip(("x", "y", "ux", "uy", "psi"), new)))

    def currents(self, s):
        opp = 1.0 + s["psi"]
        g = 1.0 / opp
        u2 = s["ux"] ** 2 + s["uy"] ** 2
        a = torch.where(s["ok"], s["q"] * s["w"], 0.0) / self.area
        return self.deposit(s["x"], s["y"], [a * (1 + u2 + opp * opp) * 0.5 * g * g, a * s["ux"] * g, a * s["uy"] * g,
                                             a * (1 + u2 - opp * opp) * 0.5 * g * g, a * s["qm"] * g])

    def beam(self, bs, i, perp=False):
        """rho, Jx, Jy, Jz (or J_perp) of the beams in slice i."""
        tot = [torch.zeros((self.ny, self.nx), **self.kw) for _ in range(2 if perp else 4)]
        for b in bs:
            k = b["sel"].get(i)
            if k is None:
                continue
            u = [b[n][k] for n in ("ux", "uy", "uz")]
            gam = torch.sqrt(1 + u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
            r = -b["w"][k] / (self.area * self.dz)
            v = [r * u[0] / gam, r * u[1] / gam] if perp else [r, r * u[0] / gam, r * u[1] / gam, r * u[2] / gam]
            tot = [t + d for t, d in zip(tot, self.deposit(b["x"][k], b["y"][k], v))]
        return tot

    def push(self, b, k, F, dt):
        x, y, z, ux, uy, uz = [b[n][k] for n in ("x", "y", "zeta", "ux", "uy", "uz")]
        h, qm = 0.5 * dt, -1.0

        def drift(x, y, z):
            ig = 1.0 / torch.sqrt(1 + ux * ux + uy * uy + uz * uz)
            return x + h * ux * ig, y + h * uy * ig, z + h * (uz * ig - 1)

        x, y, z = drift(x, y, z)
        e, f, ez, bx, by, bz = self.gather(x, y, F)
        ex, ey = e + by, f - bx
        ux, uy, uz = ux + qm * h * ex, uy + qm * h * ey, uz + qm * h * ez
        ig = 1.0 / torch.sqrt(1 + ux * ux + uy * uy + uz * uz)
        tx, ty, tz = [qm * h * t * ig for t in (bx, by, bz)]
        s = 2.0 / (1 + tx * tx + ty * ty + tz * tz)
        px, py, pz = ux + (uy * tz - uz * ty), uy + (uz * tx - ux * tz), uz + (ux * ty - uy * tx)
        ux, uy, uz = ux + s * (py * tz - pz * ty), uy + s * (pz * tx - px * tz), uz + s * (px * ty - py * tx)
        ux, uy, uz = ux + qm * h * ex, uy + qm * h * ey, uz + qm * h * ez
        x, y, z = drift(x, y, z)
        for n, v in zip(("x", "y", "zeta", "ux", "uy", "uz"), (x, y, z, ux, uy, uz)):
            b[n][k] = v

    def explicit(self, s, F4, chi, jz, bp, bn, guess):
        """(L - chi) B = rhs of the explicit solver, preconditioned conjugate gradients from `guess`."""
        e, h, ez, bz = self.gather(s["x"], s["y"], F4)
        ux, uy = s["ux"], s["uy"]
        opp = 1.0 + s["psi"]
        g = 1.0 / opp
        gam = (1 + ux * ux + uy * uy + opp * opp) * 0.5 * g
        k = -s["qm"]
        a = torch.where(s["ok"], s["q"] * s["w"], 0.0) / self.area
        dp = k * (g * (ux * e + uy * h) - ez)
        gx, gy = k * (gam * g * e + bz * g * uy), k * (gam * g * h - bz * g * ux)
        fx, fy, xx, xy, yy = self.deposit(s["x"], s["y"], [a * (g * gx - ux * g * g * dp), a * (g * gy - uy * g * g * dp),
                                                           a * g * g * ux * ux, a * g * g * ux * uy, a * g * g * uy * uy])
        tx = fx + self.ddx(xx) + self.ddy(xy) + (bp[0] - bn[0]) / (2 * self.dz)
        ty = fy + self.ddx(xy) + self.ddy(yy) + (bp[1] - bn[1]) / (2 * self.dz)
        shift = 1.0 + (1.0 / 1836.15 if self.c.get("ions") else 0.0)

        def A(v):
            p = torch.nn.functional.pad(v, (1, 1, 1, 1))
            lap = (p[1:-1, 2:] - 2 * v + p[1:-1, :-2]) / self.dx ** 2 + (p[2:, 1:-1] - 2 * v + p[:-2, 1:-1]) / self.dy ** 2
            return (chi * v - lap) * self.mask

        out = []
        for rhs, v in ((-self.ddy(jz) + ty, guess[0]), (self.ddx(jz) - tx, guess[1])):
            r = -rhs * self.mask - A(v)
            p, rz = None, None
            for _ in range(self.c["iters"]):
                z = -self.solve(r, shift)
                new = (r * z).sum()
                p = z if p is None else z + (new / rz if rz != 0 else 0.0) * p
                rz = new
                q = A(p)
                pq = (p * q).sum()
                al = rz / pq if pq != 0 else 0.0
                v, r = v + al * p, r - al * q
            out.append(v)
        return out

    def sweep(self, bs, fields=(), witness=-1, dt=0.0):
        c, n2 = self.c, (self.ny, self.nx)
        zero = torch.zeros(n2, **self.kw)
        for b in bs:
            t = torch.floor((self.zmax - b["zeta"]) / self.dz).long()
            order = torch.argsort(t)
            srt = t[order].cpu()
            b["sel"] = {}
            vals, counts = torch.unique_consecutive(srt, return_counts=True)
            at = 0
            for v, n in zip(vals.tolist(), counts.tolist()):
                if 0 <= v < self.nz:
                    b["sel"][v] = order[at:at + n]
                at += n
        s = self.plasma()
        back = zero
        if not c.get("ions"):
            back = -self.deposit(s["x"], s["y"], [s["q"] * s["w"] / self.area])[0]
        hist = [[torch.zeros_like(s["x"])] * 5 for _ in range(4)]
        b1, b2, jprev, bjprev = (zero, zero), (zero, zero), (zero, zero), (zero, zero)
        out = {k: torch.zeros((self.nz,) + n2, **self.kw) for k in fields}
        sums = [zero.sum()] * 3
        for i in range(self.nz):
            pl = self.currents(s)
            bm = self.beam(bs, i)
            rho, jx, jy, jz = [p + b for p, b in zip(pl[:4], bm)]
            rho = rho + back
            bn = self.beam(bs, i + 1, True)
            psi = self.solve(-(rho - jz))
            ez = self.solve(self.ddx(jx) + self.ddy(jy))
            bz = self.solve(self.ddy(jx) - self.ddx(jy))
            e, h = -self.ddx(psi), -self.ddy(psi)
            B = [2 * u - v for u, v in zip(b1, b2)]
            if c.get("solver", "pc") == "explicit":
                B = self.explicit(s, (e, h, ez, bz), pl[4], jz, bjprev, bn, B)
            else:
                for _ in range(c["iters"]):
                    f = self.rates(s, self.gather(s["x"], s["y"], (e, h, ez, B[0], B[1], bz)))
                    t = self.step(s, f, hist)
                    a = torch.where(t["ok"], s["q"] * s["w"], 0.0) / self.area / (1.0 + t["psi"])
                    tj = self.deposit(t["x"], t["y"], [a * t["ux"], a * t["uy"]])
                    d = [(p - q - r) / (2 * self.dz) for p, q, r in zip(jprev, tj, bn)]
                    new = (self.solve(-self.ddy(jz) + d[1]), self.solve(self.ddx(jz) - d[0]))
                    B = [MIX * u + (1 - MIX) * v for u, v in zip(new, B)]
            F = (e, h, ez, B[0], B[1], bz)
            for k, v in zip(("rho", "jx", "jy", "jz", "chi", "psi", "exmby", "eypbx", "ez", "bx", "by", "bz"),
                            (rho, jx, jy, jz, pl[4], psi, e, h, ez, B[0], B[1], bz)):
                if k in out:
                    out[k][i] = v
            if witness >= 0 and i in bs[witness]["sel"]:
                b = bs[witness]
                k = b["sel"][i]
                qw, v = -b["w"][k], self.gather(b["x"][k], b["y"][k], [ez])[0]
                sums = [t + d.sum() for t, d in zip(sums, (qw, qw * v, qw * v * v))]
            f = self.rates(s, self.gather(s["x"], s["y"], F))
            jprev, bjprev = (jx, jy), (bm[1], bm[2])
            b1, b2 = B, b1
            if dt:
                for b in bs:
                    if i in b["sel"]:
                        self.push(b, b["sel"][i], F, dt)
            s = self.step(s, f, hist)
            hist = [f] + hist[:3]
        return out, torch.stack(sums)


def exact(case, seed):
    c = case
    if c["kind"] == "solve":
        ref = _Ref(dict(c, order=1))
        return torch.stack([ref.solve(s.double()) for s in _sources(c, seed)])
    parts = c["nx"] * c["ny"] * c["ppc_x"] * c["ppc_y"] * (2 if c.get("ions") else 1) * (c["order"] + 1) ** 2
    if c["kind"] == "sweep":
        if c["nz"] * (parts * 0.2e-9 * (c["iters"] + 3) * 8 + 0.01) > 20.0:
            return None
        bs = _beams(c, seed)
        fields = c["fields"].split(",") if c["fields"] else []
        wit = 1 if c["n_witness"] else -1
        out, sums = _Ref(c).sweep(bs, fields, wit, c["dt"])
        if wit >= 0:
            out["sums"] = sums
        if c["dt"]:
            out["beams"] = [{k: b[k] for k in ("x", "y", "zeta", "ux", "uy", "uz")} for b in bs]
        return out
    if c["nz"] * parts * 8.0 * (c["iters"] + 2) * 8 > 120e9:   # the tape has to fit
        return None
    t = torch.float64 if c["precision"] == "fp64" else torch.float32
    n0 = torch.ones((), dtype=torch.float64, device="cuda", requires_grad=True)
    prof = None
    if c["profile"]:
        prof = torch.tensor(_params(c)["radial_profile"], dtype=t, device="cuda").double().requires_grad_()
    bs = _beams(c, seed)
    for b in bs:
        b["w"] = b["w"].to(t).double().requires_grad_()
    _, s = _Ref(c, n0, prof).sweep(bs, (), 1)
    loss = s[1] / s[0]
    if c["loss"] == "mean+rms":
        loss = loss + torch.sqrt(s[2] / s[0] - loss * loss)
    g = torch.autograd.grad(loss, [n0] + [b["w"] for b in bs] + ([prof] if prof is not None else []))
    return dict(loss=loss.detach(), n0=g[0], w=list(g[1:1 + len(bs)]), profile=list(g[1 + len(bs):]))
