"""The work that users of the library have it do, as measurable cases.

Each case is one pass through the public entry points of
``paper_1411_7051_gb300.lbmp`` on a lattice (or a set of lattices) that a
program holds: advancing the time loop and reading out what the study needs,
a sweep of many media, the gradient of the permeability, a new medium on an
existing lattice, the monitoring read-outs.  Sizes, drives and media are those
of the repository's configurations, tests and benchmark (the 64 x 33
validation channel, the 410 x 200 three-component medium, the 1024^2
two-component medium, the 4096^2 fractured shale, the sweep of uneven
two-component media), and generic odd ones.

``exact`` restates the method (D2Q9, Eq. 12-17 and Eq. 2 of arXiv:1411.7051)
in plain torch in 64 bits.
"""
import math

import numpy as np
import torch

from paper_1411_7051_gb300 import lbmp, media

FLOPS = 150.0        # arithmetic of one node update (moments, velocity, collision)
FLOPS_DYNAMIC = 180.0
# The stochastic rounding of FP16 sweeps draws its bits by launch shape, so a program
# whose results have to repeat pins the shape (the one that the tuner finds on the full
# sweep: the last candidate); FP32 results are the same under every shape.
STAGED_SHAPE = 9
SIDES = (256, 384, 512, 768, 1024)   # instance sides of the batched sweep


# ------------------------------------------------------------------- cases
def listed():
    return [
        # The validation channel (Section IV.A): the smallest lattice a user runs,
        # one round of the steady-state loop (100 steps, then the residual).
        dict(name="channel-64x33-fp32", kind="run", medium="channel", nx=64, ny=33, steps=100,
             storage="fp32", pressure=0, walls=1, forch=0, dyn=0, model=0, tau=0.8, read="residual"),
        # The three-component medium of Section IV.B (pores, impermeable and permeable
        # solids), with the velocity histogram of Fig. 6.
        dict(name="trimodal-410x200-fp32", kind="run", medium="trimodal", nx=410, ny=200, steps=200,
             storage="fp32", pressure=1, walls=0, forch=0, dyn=0, model=0, tau=0.9,
             read="histogram"),
        # The two-component medium at the size that inverse runs use.
        dict(name="two-component-1024-fp32", kind="run", medium="two_component", nx=1024, ny=1024,
             steps=100, storage="fp32", pressure=1, walls=1, forch=1, dyn=0, model=0, tau=0.8,
             read="permeability"),
        # The fractured shale of the benchmark, FP32 populations.
        dict(name="shale-4096-fp32", kind="run", medium="shale", nx=4096, ny=4096, steps=20,
             storage="fp32", pressure=1, walls=0, forch=1, dyn=0, model=0, tau=0.8,
             read="permeability"),
        # The same with FP16-stored populations (stochastic rounding, the default).
        dict(name="shale-4096-fp16", kind="run", medium="shale", nx=4096, ny=4096, steps=20,
             storage="fp16", pressure=1, walls=0, forch=1, dyn=0, model=0, tau=0.8,
             read="permeability"),
        # Pressure-dependent Knudsen number, ragged sizes, both storages.
        dict(name="dynamic-kn-1531x1153-fp32", kind="run", medium="shale", nx=1531, ny=1153,
             steps=50, storage="fp32", pressure=1, walls=1, forch=1, dyn=1, model=0, tau=0.8,
             read="permeability"),
        dict(name="dynamic-kn-2500x1801-fp16", kind="run", medium="shale", nx=2500, ny=1801,
             steps=30, storage="fp16", pressure=1, walls=0, forch=1, dyn=1, model=0, tau=0.8,
             read="permeability"),
        # The batched sweep of uneven media x Knudsen numbers.
        dict(name="sweep-32-fp32", kind="sweep", count=32, lo=256, hi=1024, steps=64,
             storage="fp32", walls=1),
        dict(name="sweep-32-fp16", kind="sweep", count=32, lo=256, hi=1024, steps=64,
             storage="fp16", walls=1),
        # Inverse estimation: the gradient of the permeability through the time loop.
        dict(name="gradient-1024", kind="gradient", nx=1024, ny=1024, steps=400, walls=1),
        # A new medium in pinned host memory on a lattice that is kept: set-up, a short
        # run and the permeability (the benchmark's end-to-end pass).
        dict(name="new-medium-4096-fp32", kind="medium", medium="shale", nx=4096, ny=4096, steps=20,
             storage="fp32", pressure=1, walls=0, forch=1),
        # Monitoring a running lattice: residual, mass, histogram and fields.
        dict(name="readout-4000x3001-fp32", kind="readout", medium="shale", nx=4000, ny=3001,
             storage="fp32", pressure=1, walls=0, forch=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run"] * 5 + ["sweep", "gradient", "medium", "readout"])
    storage = rng.choice(["fp32", "fp16"])
    walls = rng.randrange(2)
    if kind == "sweep":
        return dict(kind=kind, count=_log_int(rng, 4, 32), lo=rng.choice(SIDES[:3]), hi=1024,
                    steps=rng.randrange(16, 65), storage=storage, walls=walls)
    if kind == "gradient":
        nx, ny = _log_int(rng, 48, 1024), _log_int(rng, 40, 1024)
        return dict(kind=kind, nx=nx, ny=ny, steps=rng.randrange(50, 401), walls=walls)
    nx, ny = _log_int(rng, 48, 4096), _log_int(rng, 33, 4096)
    if kind == "readout":
        return dict(kind=kind, medium="shale", nx=nx, ny=ny, storage=storage, pressure=1,
                    walls=walls, forch=rng.randrange(2))
    steps = max(10, min(_log_int(rng, 10, 200), 20 * 4096 * 4096 // (nx * ny)))
    if kind == "medium":
        return dict(kind=kind, medium="shale", nx=nx, ny=ny, steps=min(steps, 20), storage=storage,
                    pressure=1, walls=walls, forch=1)
    medium = rng.choice(["channel", "two_component", "shale", "shale"])
    if medium == "channel":
        nx, ny, walls = _log_int(rng, 48, 512), _log_int(rng, 33, 257), 1
        steps = min(steps * 4, 200)
    return dict(kind=kind, medium=medium, nx=nx, ny=ny, steps=steps, storage=storage,
                pressure=0 if medium == "channel" else 1, walls=walls, forch=rng.randrange(2),
                dyn=1 if rng.random() < 0.25 else 0, model=rng.randrange(2),
                tau=rng.choice([0.7, 0.8, 0.9, 1.1]), read=rng.choice(["residual", "permeability"]))


def _sizes(case):
    """(nx, ny) of a sweep's instances: fixed by the case, uneven."""
    sides = [s for s in SIDES if case["lo"] <= s <= case["hi"]]
    r = np.random.RandomState(case["count"] * 7919 + case["lo"])
    return [(int(r.choice(sides)), int(r.choice(sides))) for _ in range(case["count"])]


# ------------------------------------------------------------------ inputs
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _generator(seed):
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _uniform(g, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device=_device(), dtype=torch.float64)


def _two_component(nx, ny, g):
    """A Gaussian random field of correlation length 32, thresholded at its median."""
    noise = torch.randn(ny, nx, generator=g, device=_device(), dtype=torch.float64)
    ky = torch.fft.fftfreq(ny, device=_device(), dtype=torch.float64)[:, None] * (2 * math.pi)
    kx = torch.fft.fftfreq(nx, device=_device(), dtype=torch.float64)[None, :] * (2 * math.pi)
    length = min(32.0, min(nx, ny) / 6.0)
    filt = torch.exp(-0.25 * (kx * kx + ky * ky) * length * length)
    field = torch.fft.ifft2(torch.fft.fft2(noise) * filt).real
    inc = field > field.median()
    eps = torch.where(inc, 0.6, 0.2).to(torch.float64)
    k_i = torch.where(inc, 1e-3, 1e-5).to(torch.float64)
    kn = torch.full_like(eps, float(_uniform(g, math.log(1e-2), math.log(10.0), 1).exp()))
    return eps, k_i, kn


def _shale(nx, ny, g):
    """A low-porosity matrix with straight fractures, Kn from the local pressure."""
    eps = _uniform(g, 0.05, 0.1, ny, nx)
    k_i = 10.0 ** (-6.0 + 0.3 * torch.randn(ny, nx, generator=g, device=_device(),
                                            dtype=torch.float64))
    r = np.random.RandomState(int(torch.randint(1 << 30, (1,), generator=g, device=_device())))
    side = math.sqrt(nx * ny)
    for _ in range(40):
        cx, cy, ang = r.uniform(0, nx), r.uniform(0, ny), r.uniform(0, math.pi)
        length, width = r.uniform(0.05, 0.5) * side, int(r.choice([2, 3, 4]))
        dx, dy = math.cos(ang), math.sin(ang)
        x0, y0 = cx - 0.5 * length * dx, cy - 0.5 * length * dy
        xa, xb = min(x0, x0 + length * dx) - width, max(x0, x0 + length * dx) + width
        ya, yb = min(y0, y0 + length * dy) - width, max(y0, y0 + length * dy) + width
        xa, xb = max(0, int(xa)), min(nx, int(xb) + 1)
        ya, yb = max(0, int(ya)), min(ny, int(yb) + 1)
        if xa >= xb or ya >= yb:
            continue
        px = torch.arange(xa, xb, device=_device(), dtype=torch.float64)[None, :] - x0
        py = torch.arange(ya, yb, device=_device(), dtype=torch.float64)[:, None] - y0
        t = (px * dx + py * dy).clamp(0.0, length)
        mask = (px - t * dx) ** 2 + (py - t * dy) ** 2 <= (0.5 * width) ** 2
        eps[ya:yb, xa:xb].masked_fill_(mask, 0.9)
        k_i[ya:yb, xa:xb].masked_fill_(mask, 1e-2)
    x = torch.arange(nx, device=_device(), dtype=torch.float64) / max(nx - 1, 1)
    kn = 0.5 / (1.0 - 0.5 * x)[None, :] * math.sqrt(1e-6 / 0.075) / (k_i / eps).sqrt()
    return eps, k_i, kn


def _fields(case, seed):
    """Porosity, intrinsic permeability and Knudsen number, [ny, nx] float64."""
    nx, ny = case["nx"], case["ny"]
    g = _generator(seed)
    name = case.get("medium", "two_component")
    if name == "two_component":
        return _two_component(nx, ny, g)
    if name == "shale":
        return _shale(nx, ny, g)
    if name == "trimodal":
        lab = media.trimodal(nx, ny, seed=int(seed) % (1 << 31))
        m = media.trimodal_medium(lab, 0.3, 1e-2, 0.38)
        return tuple(torch.from_numpy(a).to(_device()) for a in (m.eps, m.k_i, m.kn))
    gap = ny - 2
    shape = (ny, nx)
    eps = torch.full(shape, 0.7, device=_device(), dtype=torch.float64)
    k_i = torch.full(shape, 1e-3 * gap * gap, device=_device(), dtype=torch.float64)
    k_i *= torch.exp(0.2 * torch.randn(shape, generator=g, device=_device(), dtype=torch.float64))
    return eps, k_i, torch.full_like(eps, float(_uniform(g, 0.02, 0.5, 1)))


def _config(case, seed, nx, ny):
    pressure = case.get("pressure", 1)
    return lbmp.SimConfig(
        nx, ny, tau=case.get("tau", 0.8), G=(0.0, 0.0) if pressure else (1e-6, 0.0),
        bc_x=lbmp.BCX_PRESSURE if pressure else lbmp.BCX_PERIODIC,
        bc_y=lbmp.BCY_WALLS if case["walls"] else lbmp.BCY_PERIODIC,
        rho_in=1.0005 if pressure else 1.0, rho_out=0.9995 if pressure else 1.0,
        forchheimer=case.get("forch", 1),
        storage=lbmp.STORE_FP16 if case.get("storage") == "fp16" else lbmp.STORE_FP32,
        kn_model=case.get("model", 0), kn_beta=_kn_beta(case), seed=int(seed))


def _kn_beta(case):
    """The inlet pressure is twice the outlet one (rho 1.0005 -> 0.9995)."""
    return 1.0 / 1.5e-3 if case.get("dyn") and case.get("pressure", 1) else 0.0


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        sizes = _sizes(case)
        batch = lbmp.Batch(_config(case, seed, 1, 1), sizes)
        for i, (nx, ny) in enumerate(sizes):
            batch.set_fields(i, *_fields(dict(case, nx=nx, ny=ny), seed * 1009 + i))
        if case["storage"] == "fp16":
            batch.set_shape(STAGED_SHAPE)
        else:
            batch.tune_cached(steps=4)
        return dict(case=case, batch=batch)
    sim = lbmp.Sim(_config(case, seed, case["nx"], case["ny"]))
    eps, k_i, kn = _fields(case, seed)
    if kind == "gradient":
        return dict(case=case, sim=sim, kn=kn, log_k=k_i.log().requires_grad_(True),
                    eps=eps.requires_grad_(True))
    if kind == "medium":
        return dict(case=case, sim=sim, fields=[t.cpu().pin_memory() for t in (eps, k_i, kn)])
    sim.set_fields(eps, k_i, kn)
    if kind == "readout":
        sim.step(20)
    return dict(case=case, sim=sim)


# --------------------------------------------------------------------- run
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "sweep":
        batch = state["batch"]
        batch.step(case["steps"])
        kg, um = batch.permeability()
        return [kg, um] + [batch.populations(i) for i in range(batch.count)]
    sim = state["sim"]
    if kind == "gradient":
        log_k, eps = state["log_k"], state["eps"]
        kg = lbmp.ka_from_fields(sim, log_k, eps, state["kn"], case["steps"])
        d_logk, d_eps = torch.autograd.grad(kg, (log_k, eps))
        return [kg.detach(), d_logk, d_eps]
    if kind == "readout":
        residual = sim.residual()
        counts, umax = sim.velocity_histogram(10)
        return [residual, sim.mass(), counts, umax, *sim.permeability(), *sim.macroscopic(),
                sim.apparent_permeability()]
    if kind == "medium":
        sim.set_fields(*state["fields"])
        sim.step(case["steps"])
        return [*sim.permeability(), *sim.macroscopic()]
    sim.step(case["steps"])
    out = [*sim.permeability()]
    if case["read"] == "residual":
        out.append(sim.residual())
    if case["read"] == "histogram":
        counts, umax = sim.velocity_histogram(10)
        out += [counts, umax]
    return out + [*sim.macroscopic()]


# -------------------------------------------------------------------- work
def work(case):
    """The populations and the medium read once, the populations and the
    outputs written once; the arithmetic of every node update."""
    kind = case["kind"]
    elem = 2 if case.get("storage") == "fp16" else 4
    flops = FLOPS_DYNAMIC if case.get("dyn") and case.get("pressure", 1) else FLOPS
    if kind == "sweep":
        nodes = sum(nx * ny for nx, ny in _sizes(case))
        return dict(bytes=nodes * (18.0 * elem + 8.0 + 72.0), flops=nodes * flops * case["steps"])
    nodes = float(case["nx"] * case["ny"])
    if kind == "gradient":  # the medium in, two gradients out; forward and backward per step
        return dict(bytes=nodes * 40.0, flops=nodes * 3.0 * flops * case["steps"])
    if kind == "readout":   # one read of the state, velocity snapshot in and out, four fields out
        return dict(bytes=nodes * (9.0 * elem + 8.0 + 16.0 + 32.0), flops=nodes * 60.0)
    if kind == "medium":
        return dict(bytes=nodes * (24.0 + 9.0 * elem + 8.0 + 24.0),
                    flops=nodes * flops * case["steps"])
    return dict(bytes=nodes * (18.0 * elem + 8.0 + 24.0), flops=nodes * flops * case["steps"])


# ------------------------------------------------- the method in 64 bits
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


class _Exact:
    def __init__(self, cfg, eps, k_i, kn):
        self.cfg, self.eps = cfg, eps
        self.nu = (cfg.tau - 0.5) / 3.0 / cfg.J
        self.walls = cfg.bc_y == lbmp.BCY_WALLS
        self.pressure = cfg.bc_x == lbmp.BCX_PRESSURE
        self.k_i, self.kn = k_i, kn
        self.inv_ka = None if cfg.kn_beta else 1.0 / (k_i * self.fc(kn))
        self.solid = eps == 0.0
        self.any_solid = bool(self.solid.any())
        self.safe = torch.where(self.solid, 1.0, eps) if self.any_solid else eps
        self.rows = slice(1, -1) if self.walls else slice(None)

    def fc(self, kn):
        if self.cfg.kn_model == lbmp.KN_FIRST_ORDER:
            return 1.0 + 4.0 * kn
        alpha = 1.358 / (1.0 + 0.170 * kn ** -0.4348)
        return (1.0 + alpha * kn) * (1.0 + 4.0 * kn / (1.0 + kn))

    def rest(self):
        w = torch.tensor(W, device=self.eps.device, dtype=torch.float64).view(9, 1, 1)
        return self.extrapolate((w * self.cfg.rho0).expand(9, *self.eps.shape).clone())

    def state(self, f, cut=None):
        """Density, velocity and force of every node (or of the columns ``cut``)."""
        c = self.cfg
        at = (lambda t: t) if cut is None else (lambda t: t[:, cut])
        eps, solid = at(self.safe), at(self.solid)
        rho = f.sum(0)
        mx = f[1] - f[3] + f[5] - f[6] - f[7] + f[8]
        my = f[2] - f[4] + f[5] + f[6] - f[7] - f[8]
        if c.kn_beta:
            q = 1.0 + c.kn_beta * (rho - c.rho0)
            inv = 1.0 / (at(self.k_i) * self.fc(at(self.kn) / q))
        else:
            inv = at(self.inv_ka)
        vx = mx / rho + 0.5 * eps * c.G[0]
        vy = my / rho + 0.5 * eps * c.G[1]
        darcy = eps * self.nu * inv
        c0 = 0.5 * (1.0 + 0.5 * darcy)
        if c.forchheimer:
            c1 = 0.5 * eps * (1.75 / (150.0 * eps ** 3).sqrt()) * inv.sqrt()
            v2 = vx * vx + vy * vy
            zero = v2 == 0.0
            vmag = torch.where(zero, torch.zeros_like(v2), torch.where(zero, 1.0, v2).sqrt())
            den = c0 + (c0 * c0 + c1 * vmag).sqrt()
            drag = darcy + 2.0 * c1 * vmag / den
        else:
            den, drag = 2.0 * c0, darcy
        ux, uy = vx / den, vy / den
        fx, fy = eps * c.G[0] - drag * ux, eps * c.G[1] - drag * uy
        if self.any_solid:
            ux, uy = torch.where(solid, 0.0, ux), torch.where(solid, 0.0, uy)
            fx, fy = torch.where(solid, -2.0 * mx / rho, fx), torch.where(solid, -2.0 * my / rho, fy)
        return rho, ux, uy, fx, fy, eps

    @staticmethod
    def feq(i, rho, ux, uy, eps):
        eu = EX[i] * ux + EY[i] * uy
        return W[i] * rho * (1.0 + 3.0 * eu + (4.5 * eu * eu - 1.5 * (ux * ux + uy * uy)) / eps)

    def collide(self, f):
        rho, ux, uy, fx, fy, eps = self.state(f)
        tau, out = self.cfg.tau, []
        uf = ux * fx + uy * fy
        for i in range(9):
            eu, ef = EX[i] * ux + EY[i] * uy, EX[i] * fx + EY[i] * fy
            force = W[i] * rho * (1.0 - 0.5 / tau) * (3.0 * ef + (9.0 * eu * ef - 3.0 * uf) / eps)
            out.append(f[i] - (f[i] - self.feq(i, rho, ux, uy, eps)) / tau + force)
        return out

    def extrapolate(self, f):
        if not self.pressure:
            return f
        nx, new = f.shape[2], []
        for b, n, rho_b in ((0, 1, self.cfg.rho_in), (nx - 1, nx - 2, self.cfg.rho_out)):
            fn = f[:, :, n:n + 1]
            rho, ux, uy, _, _, eps_n = self.state(fn, slice(n, n + 1))
            eps_b, solid_b = self.safe[:, b:b + 1], self.solid[:, b:b + 1]
            bx, by = torch.where(solid_b, 0.0, ux), torch.where(solid_b, 0.0, uy)
            new.append(torch.stack([self.feq(i, rho_b * torch.ones_like(rho), bx, by, eps_b)
                                    + fn[i] - self.feq(i, rho, ux, uy, eps_n)
                                    for i in range(9)]))
        return torch.cat([new[0], f[:, :, 1:-1], new[1]], 2)

    def step(self, f):
        post, out = self.collide(f), []
        for i in range(9):
            g = torch.roll(post[i], (EY[i], EX[i]), (0, 1))
            if self.walls and EY[i]:
                y = 1 if EY[i] > 0 else g.shape[0] - 2   # the source row is a plate
                back = post[OPP[i]][y:y + 1]
                g = torch.cat([g[:y], back, g[y + 1:]], 0)
            out.append(g)
        return self.extrapolate(torch.stack(out))

    def read(self, f):
        rho, ux, uy = (t.clone() for t in self.state(f)[:3])
        if self.walls:
            for t in (rho, ux, uy):
                t[0] = 0.0
                t[-1] = 0.0
        return rho, ux, uy

    def permeability(self, ux):
        c, g = self.cfg, self.cfg.G[0]
        um = ux[self.rows].mean()
        if self.pressure:
            g = g + (c.rho_in - c.rho_out) / 3.0 / self.eps[self.rows].mean() / (
                c.rho0 * (self.eps.shape[1] - 1))
        return self.nu * um / g, um


def _exact_run(case, seed, steps):
    cfg = _config(case, seed, case["nx"], case["ny"])
    e = _Exact(cfg, *_fields(case, seed))
    f = e.rest()
    for _ in range(steps):
        f = e.step(f)
    return e, f


def _exact_gradient(case, seed):
    from torch.utils.checkpoint import checkpoint
    cfg = _config(case, seed, case["nx"], case["ny"])
    eps, k_i, kn = _fields(case, seed)
    log_k = k_i.log().requires_grad_(True)
    eps.requires_grad_(True)

    def advance(f, log_k, eps, n):
        e = _Exact(cfg, eps, log_k.exp(), kn)
        for _ in range(n):
            f = e.step(f)
        return f

    f = _Exact(cfg, eps, log_k.exp(), kn).rest()
    left = case["steps"]
    while left:
        n = min(20, left)
        f = checkpoint(advance, f, log_k, eps, n, use_reentrant=False)
        left -= n
    e = _Exact(cfg, eps, log_k.exp(), kn)
    kg, _ = e.permeability(e.state(f)[1])
    d_logk, d_eps = torch.autograd.grad(kg, (log_k, eps))
    for t in (d_logk, d_eps):
        if cfg.bc_y == lbmp.BCY_WALLS:
            t[0] = 0.0
            t[-1] = 0.0
    return [kg.detach(), d_logk, d_eps]


def exact(case, seed):
    kind = case["kind"]
    if kind == "gradient":
        return _exact_gradient(case, seed)
    with torch.no_grad():
        if kind == "sweep":
            kgs, ums, pops = [], [], []
            for i, (nx, ny) in enumerate(_sizes(case)):
                one = dict(case, nx=nx, ny=ny)
                e = _Exact(_config(case, seed, nx, ny), *_fields(one, seed * 1009 + i))
                f = e.rest()
                for _ in range(case["steps"]):
                    f = e.step(f)
                kg, um = e.permeability(e.state(f)[1])
                if e.walls:
                    f[:, 0] = 0.0
                    f[:, -1] = 0.0
                kgs.append(float(kg))
                ums.append(float(um))
                pops.append(f)
            return [np.array(kgs), np.array(ums)] + pops
        if kind == "readout":
            e, f = _exact_run(case, seed, 20)
            rho, ux, uy = e.read(f)
            kg, um = e.permeability(ux)
            ka = e.k_i * e.fc(e.kn)
            if e.walls:
                ka[0] = 0.0
                ka[-1] = 0.0
            # the snapshot before the first residual is zero: the residual is 1
            return [1.0, float(rho[e.rows].sum()), None, float((ux * ux + uy * uy).max().sqrt()),
                    float(kg), float(um), rho, ux, uy, ka]
        e, f = _exact_run(case, seed, case["steps"])
        rho, ux, uy = e.read(f)
        kg, um = e.permeability(ux)
        out = [float(kg), float(um)]
        if kind == "run" and case["read"] == "residual":
            out.append(1.0)
        if kind == "run" and case["read"] == "histogram":
            out += [None, float((ux * ux + uy * uy).max().sqrt())]
        return out + [rho, ux, uy]
