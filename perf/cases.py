"""Performance cases of the D2Q9 library: what its users run, through the public entry points.

Every case is one call of a simulation loop: advance the context by ``steps`` timesteps
(``Context.step``), write the density and velocity fields into device tensors
(``Context.moments_device``) and, where there are particles, receive their state after
every step in page-locked host memory (``Context.record_particles``).  The contexts, with
the graphs of the repeated step count (``prepare_steps``), are made once, as a program
that simulates for hours makes them.

The workloads are those of ``paper_2006_12910_gb300/workloads.py`` (the configurations of
the benchmark and of the tests) at their own sizes, from one 128x128 domain to ten million
nodes, with every storage kind and option in use.  ``draw`` varies sizes (odd widths and
heights among them), step counts, storage kinds, relaxation times and options.
"""
import functools
import math

import numpy as np
import torch

from paper_2006_12910_gb300 import lbm, workloads

HALF_SCALE = 4096.0  # power-of-two scale of the shifted half-precision stores
STORE_BYTES = {"f64": 8, "f32": 4, "f32s": 4, "f16s": 2, "bf16s": 2}
MAX_NODES = 4096 * 2048
FIELDS = dict(kind="", nx=0, ny=0, store="f32s", steps=20, particles=0, n_pl=0.0, tau=0.0, domains=0)


def _case(name=None, **kw):
    c = dict(FIELDS, **kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smooth BGK channel of the convergence study: a small lattice in FP64, many steps per call
        _case("channel_256x64_f64", kind="channel", nx=256, ny=64, store="f64", steps=100, tau=0.8),
        # one realisation of the smallest ensemble size, observed after every step: the smallest call
        _case("flb_128_one_step", kind="flb", nx=128, ny=128, steps=1, particles=1),
        # Brownian disk in the narrow walled channel of the paper's second benchmark (odd height, ragged width)
        _case("brownian_3000x41", kind="brownian", nx=3000, ny=41, steps=20, particles=1),
        # fluctuating fluid with one Brownian disk, the equipartition study
        _case("flb_512", kind="flb", nx=512, ny=512, steps=20, particles=1),
        # pseudoplastic fluid: local relaxation time at every node
        _case("power_law_4096x256", kind="channel", nx=4096, ny=256, steps=20, n_pl=0.75),
        # flow through grains in the shape of the paper's first benchmark, 45 disks, periodic along x, ragged width
        _case("grains_1620x1020", kind="grains", nx=1620, ny=1020, steps=20, particles=45),
        # the benchmark workload: fractured porous domain, open ends, 20 free disks ...
        _case("porous_2048x1024", kind="porous", nx=2048, ny=1024, steps=20, particles=20, tau=0.7),
        # ... with the half-precision store that fits twice the lattice in memory
        _case("porous_2048x1024_f16s", kind="porous", nx=2048, ny=1024, store="f16s", steps=2, particles=20, tau=0.7),
        # ... and as the FP64 reference run
        _case("porous_2048x1024_f64", kind="porous", nx=2048, ny=1024, store="f64", steps=4, particles=20, tau=0.7),
        # every feature at once: obstacles, particles, open ends, noise and a power-law fluid
        _case("combined_2048x1024", kind="combined", nx=2048, ny=1024, steps=10, particles=20, n_pl=1.5, tau=0.7),
        # 96 uneven fluctuating domains with a Brownian disk each, advanced together (10 million nodes)
        _case("ensemble_96", kind="ensemble", steps=20, particles=1, domains=96),
        # the largest single lattice: permeability run through the rock alone, no particles
        _case("porous_4096x2048", kind="porous", nx=4096, ny=2048, steps=10, tau=0.7),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["channel", "channel", "flb", "brownian", "grains", "porous", "porous", "combined", "ensemble"])
    tau = round(rng.uniform(0.6, 1.2), 3)
    store = rng.choice(["f32s", "f32s", "f32s", "f32", "f64", "f16s", "bf16s"])
    steps = _log_int(rng, 1, 32)
    if store in ("f16s", "bf16s"):  # one output step between observations: the store's rounding is what a user looks at
        steps = rng.choice([1, 2])
    if kind == "channel":
        nx, ny = _log_int(rng, 96, 6000), _log_int(rng, 32, 512)
        n_pl = rng.choice([0.0, 0.0, 0.5, 0.75, 1.5])
        if n_pl and store in ("f16s", "bf16s"):
            store = "f32s"
        return _case(kind=kind, nx=nx, ny=ny, store=store, steps=4 * steps if nx * ny < 100000 else steps, n_pl=n_pl,
                     tau=tau if not n_pl else 0.0)
    if store == "f64" or kind not in ("porous",):
        store = "f64" if store == "f64" and kind in ("porous", "flb") else "f32s"
    if kind == "flb":
        return _case(kind=kind, nx=_log_int(rng, 100, 1000), ny=_log_int(rng, 100, 1000), store=store, steps=steps,
                     particles=1)
    if kind == "brownian":
        return _case(kind=kind, nx=_log_int(rng, 400, 6000), ny=rng.randrange(33, 90), steps=steps, particles=1)
    if kind == "grains":
        return _case(kind=kind, nx=_log_int(rng, 700, 2400), ny=_log_int(rng, 300, 1200), steps=steps, particles=45)
    if kind == "ensemble":
        return _case(kind=kind, steps=steps, particles=1, domains=rng.randrange(4, 96))
    nx = _log_int(rng, 400, 3000)
    ny = max(300, min(_log_int(rng, 300, 2000), 3000 * 1500 // nx))
    if kind == "combined":
        return _case(kind=kind, nx=nx, ny=ny, steps=min(steps, 12), particles=rng.randrange(1, 24), n_pl=1.5, tau=tau)
    return _case(kind=kind, nx=nx, ny=ny, store=store, steps=min(steps, 6) if store == "f64" else steps,
                 particles=rng.choice([0, 1, 8, 20]), tau=tau)


# ---------------------------------------------------------------------------------------
# Workloads: geometry and particles by size (a user's program has them before the first
# call), initial populations and noise key by seed.
# ---------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=8)
def _workload(kind, nx, ny, particles, n_pl, tau, domains):
    """[(nx, ny, params, solid or None, particle dicts)] of the case's domains."""
    if kind == "channel":
        if n_pl:
            w = workloads.power_law(n_pl, nx, ny, g=2e-8 if n_pl > 1 else 1e-6)
        else:
            w = workloads.poiseuille(nx, ny)
            w.params["tau"] = tau
        ws = [w]
    elif kind == "flb":
        ws = [workloads.flb(nx, ny)]
    elif kind == "brownian":
        ws = [workloads.confined_channel(nx, ny)]
    elif kind == "grains":
        ws = [workloads.grains(nx, ny, n_obstacles=max(1, round(236 * nx * ny / (1620 * 1020))))]
    elif kind == "porous":
        ws = [workloads.porous(nx, ny, n_particles=0)]
    elif kind == "combined":
        ws = [workloads.combined(nx, ny, n_pl=n_pl)]
    else:
        ws = workloads.ensemble(domains)
    if kind in ("porous", "combined"):
        w = ws[0]
        w.params["tau"] = tau
        disks = workloads.place_obstacles(nx, ny, max(1, round(300 * nx * ny / (2048 * 1024))), 8.0, 24.0, gap=4.0,
                                          margin_y=2.0, margin_x=6.0, seed=workloads.BASE_SEED + 2)
        w.particles = workloads.place_particles(nx, ny, particles, 10.0, 1.05, disks, gap=4.5, margin_y=2.0,
                                                x_range=(0.1 * nx, 0.6 * nx), seed=workloads.BASE_SEED + 1002) \
            if particles else []
    return [(w.nx, w.ny, w.params, w.solid, w.particles) for w in ws]


def _domains(case):
    return _workload(case["kind"], case["nx"], case["ny"], case["particles"], case["n_pl"], case["tau"],
                     case["domains"])


def _populations(case, seed, dom, nx, ny, params, solid):
    """Initial f[9][ny][nx] on the GPU in FP64: a flow with large-scale structure and, in the
    channels, a developed profile; the amplitude is that of the thermal velocities where
    there is noise."""
    g = torch.Generator(device="cuda").manual_seed(1000003 * (seed + 1) + dom)
    kw = dict(device="cuda", dtype=torch.float64)
    a = torch.rand(9, 4, generator=g, **kw).tolist()
    y, x = torch.arange(ny, **kw)[:, None], torch.arange(nx, **kw)[None, :]
    if case["kind"] == "channel":
        # a shear flow like the developed one, with a weak variation along the channel and a weak cross flow
        n = case["n_pl"] or 1.0
        s = (2.0 * (y + 0.5) / ny - 1.0).abs()
        u = (0.01 + 0.02 * a[0][0]) * (1.0 - s ** ((n + 1.0) / n)) * (1 + 0.01 * torch.sin(2 * math.pi * (x / nx + a[0][1])))
        v = (0.002 + 0.004 * a[0][3]) * (1.0 - s * s) * torch.sin(2 * math.pi * (x / nx + a[1][0]))
        r = 1.0 + 1e-4 * torch.cos(2 * math.pi * (x / nx + a[0][2])) * torch.ones_like(u)
        f = torch.empty(9, ny, nx, **kw)
        for i in range(9):
            eu = 3.0 * (EX[i] * u + EY[i] * v)
            f[i] = WGT[i] * r * (1.0 + eu + 0.5 * eu * eu - 1.5 * (u * u + v * v))
        return f
    amp = 0.003 if params.get("kT", 0.0) > 0 else 0.01
    f = torch.randn(9, ny, nx, generator=g, **kw).mul_(0.5)
    for i in range(9):
        kx, ky = 1 + int(3 * a[i][0]), 1 + int(3 * a[i][1])
        f[i] += torch.sin(2 * math.pi * (kx * x / nx + ky * y / ny + a[i][2]))
        f[i].mul_(amp * WGT[i]).add_(WGT[i])
    if solid is not None:
        f[:, torch.from_numpy(solid).cuda() != 0] = 0.0
    return f


def _seeded(params, seed, dom):
    p = dict(params)
    if p.get("kT", 0.0) > 0:
        p["seed"] = (p["seed"] + 7919 * (seed + 1)) % (1 << 63)
    return p


class _State:
    pass


def prepare(case, seed):
    doms = _domains(case)
    s = _State()
    s.stream = torch.cuda.Stream()
    scale = HALF_SCALE if case["store"] in ("f16s", "bf16s") else 1.0
    prm = [lbm.make_params(nx=nx, ny=ny, store=case["store"], store_scale=scale, max_particles=len(parts),
                           **_seeded(params, seed, d)) for d, (nx, ny, params, _, parts) in enumerate(doms)]
    s.ctx = lbm.Context(prm, stream=s.stream, solids=[d[3] for d in doms])
    for d, (nx, ny, params, solid, parts) in enumerate(doms):
        s.ctx.set_populations(_populations(case, seed, d, nx, ny, params, solid).cpu().numpy(), dom=d)
        if parts:
            s.ctx.add_particles(d, parts)
    s.out = {k: torch.zeros(sum(d[0] * d[1] for d in doms), device="cuda") for k in ("rho", "ux", "uy")}
    s.views, at = [], 0
    for nx, ny, *_ in doms:
        s.views.append([t[at:at + nx * ny] for t in s.out.values()])
        at += nx * ny
    if s.ctx.particle_slots:
        s.out["particles"] = torch.zeros(case["steps"], s.ctx.particle_slots, 6, dtype=torch.float64, pin_memory=True)
        s.ctx.record_particles(s.out["particles"])
    s.steps = case["steps"]
    s.ctx.prepare_steps(s.steps)
    return s


def run(state):
    state.ctx.step(state.steps)
    for d, v in enumerate(state.views):
        state.ctx.moments_device(*v, dom=d)
    return state.out


def work(case):
    """Per step every fluid node reads and writes its nine populations once; then the fields
    are formed from one read of the populations.  Operations per node and step: the BGK
    collision (75), noise (two Philox4x32-10 blocks, six normals, the projection: 330) and
    the local relaxation time (about six Newton steps: 90)."""
    b = f = 0
    s = STORE_BYTES[case["store"]]
    for nx, ny, params, solid, parts in _domains(case):
        fluid = nx * ny - (int(solid.sum()) if solid is not None else 0)
        b += case["steps"] * 18 * s * fluid + 9 * s * fluid + 12 * nx * ny + case["steps"] * 48 * len(parts)
        f += case["steps"] * fluid * (75 + (330 if params.get("kT", 0.0) > 0 else 0) + (90 if params.get("power_law") else 0))
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------------------
# The same in 64 bits, as plain tensor operations (arXiv:2006.12910 Secs. 2-5).
# ---------------------------------------------------------------------------------------
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
WGT = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
M32 = 0xFFFFFFFF


def _philox(ctr, k0, k1):
    """Philox4x32-10 (Salmon et al. 2011) on int64 tensors holding 32-bit words."""
    c0, c1, c2, c3 = ctr
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57  # low 64 bits; the shifts below take them as unsigned
        c0, c1, c2, c3 = ((p1 >> 32) & M32) ^ c1 ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c3 ^ k1, p0 & M32
    return c0, c1, c2, c3


def _normals(node, step, dom, k0, k1):
    out = []
    for d in (0, 1):
        z = torch.zeros_like(node)
        w = [((v >> 9).double() + 0.5) / 8388608.0 for v in _philox((node + z, z + step, z + d, z + dom), k0, k1)]
        for u, v in ((w[0], w[1]), (w[2], w[3]))[:2 - d]:
            r = torch.sqrt(-2.0 * torch.log(u))
            out += [r * torch.cos(2 * math.pi * v), r * torch.sin(2 * math.pi * v)]
    return out


def _mode(k, i):
    e2 = EX[i] ** 2 + EY[i] ** 2
    v, w = {3: (3 * e2 - 2, 4), 4: (2 * EX[i] ** 2 - e2, 4 / 9), 5: (EX[i] * EY[i], 1 / 9),
            6: ((3 * e2 - 4) * EX[i], 2 / 3), 7: ((3 * e2 - 4) * EY[i], 2 / 3), 8: (9 * e2 * e2 - 15 * e2 + 2, 16)}[k]
    return v / math.sqrt(w)


class _Exact:
    """Domains of one size in FP64, f[9][domain][ny][nx], post-collision populations."""

    def __init__(self, nx, ny, params, solid, f, parts):
        self.nx, self.ny, self.f, self.t = nx, ny, f, 0
        self.p = {k: params[0].get(k, 0) for k in ("periodic_x", "periodic_y", "tau", "gx", "gy", "rho_in", "rho_out",
                                                   "power_law", "n_pl", "xi_pl", "tau_min", "tau_max", "lj_psi", "lj_rit",
                                                   "inlet_outlet")}
        dev = f.device
        col = lambda key, kind: torch.tensor([p.get(key, 0) for p in params], device=dev, dtype=kind)[:, None, None]  # noqa: E731
        self.kT, self.dom = col("kT", torch.float64), col("domain_id", torch.int64)
        self.k0 = torch.tensor([int(p.get("seed", 0)) & M32 for p in params], device=dev)[:, None, None]
        self.k1 = torch.tensor([int(p.get("seed", 0)) >> 32 for p in params], device=dev)[:, None, None]
        self.node = torch.arange(nx * ny, device=dev).view(1, ny, nx)
        self.solid = torch.zeros(ny, nx, dtype=torch.bool, device=dev) if solid is None else torch.from_numpy(solid).to(dev) != 0
        # where direction i comes from a solid or from beyond a wall (or, on wall rows, an open end): bounced back
        y, x = torch.arange(ny, device=dev)[:, None], torch.arange(nx, device=dev)[None, :]
        self.bounce, self.any_bounce = [], []
        for i in range(9):
            b = torch.roll(self.solid, (EY[i], EX[i]), (0, 1))
            if not self.p["periodic_y"]:
                b = b | (y - EY[i] < 0) | (y - EY[i] >= ny)
            if self.p["inlet_outlet"]:
                outside = (x - EX[i] < 0) | (x - EX[i] >= nx)
                b = (b & ~outside) | (outside & ((y == 0) | (y == ny - 1)))
            self.bounce.append(b)
            self.any_bounce.append(bool(b.any()))
        flat = [(d, q) for d, ps in enumerate(parts) for q in ps]
        self.np = len(flat)
        if self.np:
            get = lambda key: torch.tensor([float(q.get(key, 0.0)) for _, q in flat], device=dev, dtype=torch.float64)  # noqa: E731
            self.pd = torch.tensor([d for d, _ in flat], device=dev)
            self.R, self.rho_p = get("R"), get("rho_p")
            self.X = torch.stack([get(k) for k in ("x", "y", "U", "V", "Omega", "theta")], 1)
            self.m = self.rho_p * math.pi * self.R ** 2
            self.I = 0.5 * self.m * self.R ** 2
            self.prev = self.X[:, :2].clone()

    def gather(self, node, ok):
        """(flat index, valid) of unwrapped nodes (y, x) [np, h, w]."""
        y, x = node
        if self.p["periodic_y"]:
            y = y % self.ny
        else:
            ok = ok & (y >= 0) & (y < self.ny)
        if self.p["periodic_x"]:
            x = x % self.nx
        else:
            ok = ok & (x >= 0) & (x < self.nx)
        y, x = y.clamp(0, self.ny - 1), x.clamp(0, self.nx - 1)
        return (self.pd[:, None, None] * self.ny + y) * self.nx + x, ok

    def image(self, d, axis):
        n = self.nx if axis == 0 else self.ny
        return d - n * torch.round(d / n) if self.p["periodic_x" if axis == 0 else "periodic_y"] else d

    def inside(self, c, y, x):
        """Strictly inside the disks of centres c, nodes (y, x) unwrapped near them."""
        dx, dy = self.image(x - c[:, 0, None, None], 0), self.image(y - c[:, 1, None, None], 1)
        return dx * dx + dy * dy < (self.R ** 2)[:, None, None]

    def repulsion(self, y, x, ax, ay, ins):
        """Eq. MP2 between surface nodes of a disk and those of others, solids and walls."""
        p, surf = self.p, torch.zeros_like(ins)
        c = self.X[:, :2]
        for i in range(1, 9):
            surf |= ins & ~self.inside(c, y + EY[i], x + EX[i])
        idx, ok = self.gather((y, x), torch.ones_like(surf))
        count = torch.zeros(self.f[0].numel(), dtype=torch.float64, device=self.f.device)
        count.index_put_((idx[surf & ok],), torch.ones((), dtype=torch.float64, device=count.device), accumulate=True)
        F = torch.zeros(self.np, 3, dtype=torch.float64, device=count.device)
        reach = int(p["lj_rit"])
        for oy in range(-reach, reach + 1):
            for ox in range(-reach, reach + 1):
                dist = math.hypot(ox, oy)
                if not 0 < dist <= p["lj_rit"]:
                    continue
                mag = p["lj_psi"] * (dist / p["lj_rit"]) ** -13.0
                jdx, jok = self.gather((y + oy, x + ox), torch.ones_like(surf))
                own = self.inside(c, y + oy, x + ox)
                edge = torch.zeros_like(own)
                for i in range(1, 9):
                    edge |= own & ~self.inside(c, y + oy + EY[i], x + ox + EX[i])
                wall = torch.zeros_like(surf) if p["periodic_y"] else (y + oy < 0) | (y + oy >= self.ny)
                wall = (wall | (jok & self.solid.view(-1)[jdx % (self.ny * self.nx)])) & ok & ~self.solid.view(-1)[idx % (self.ny * self.nx)]
                hits = surf * (wall.double() + jok * (count[jdx] - edge.double()))
                fx, fy = -mag * ox / dist * hits, -mag * oy / dist * hits
                F += torch.stack([fx.sum((1, 2)), fy.sum((1, 2)), (ax * fy - ay * fx).sum((1, 2))], 1)
        return F

    def move_particles(self):
        """Forces at t, Newton-Euler and the link exchange (Eqs. MP1-MP8) on f."""
        p, f, dev = self.p, self.f.view(9, -1), self.f.device
        c, R = self.X[:, :2].clone(), self.R
        h = int(math.ceil(float(R.max()))) + 6
        o = torch.arange(-h, h + 1, device=dev)
        y, x = (torch.floor(c[:, 1]).long()[:, None, None] + o[:, None]), (torch.floor(c[:, 0]).long()[:, None, None] + o[None, :])
        y, x = y.expand(-1, -1, 2 * h + 1), x.expand(-1, 2 * h + 1, -1)
        idx, ok = self.gather((y, x), torch.ones_like(y, dtype=torch.bool))
        fluid = ok & ~self.solid.view(-1)[idx % (self.ny * self.nx)]
        ins = self.inside(c, y, x)
        covered = torch.zeros(f.shape[1], dtype=torch.bool, device=dev)
        covered[idx[ins & ok]] = True
        ax, ay = x - c[:, 0, None, None], y - c[:, 1, None, None]  # arms of the nodes
        G = torch.zeros(self.np, 3, dtype=torch.float64, device=dev)
        Z = torch.zeros(self.np, 3, 3, dtype=torch.float64, device=dev)
        links = []
        for k in range(1, 9):
            jdx, jok = self.gather((y + EY[k], x + EX[k]), fluid)
            link = ins & fluid & jok & ~self.solid.view(-1)[jdx % (self.ny * self.nx)] & ~covered[jdx]
            w, n, j = torch.nonzero(link)[:, 0], idx[link], jdx[link]
            arm = (ax[link] + 0.5 * EX[k]) * EY[k] - (ay[link] + 0.5 * EY[k]) * EX[k]
            a = torch.stack([torch.full_like(arm, EX[k]), torch.full_like(arm, EY[k]), arm], 1)
            G.index_add_(0, w, -2.0 * f[OPP[k]][j][:, None] * a)
            Z.index_add_(0, w, 6.0 * WGT[k] * a[:, :, None] * a[:, None, :])
            links.append((k, w, n, j, a))
        was = self.inside(self.prev, y, x)
        flip = fluid & (was != ins)
        w, n = torch.nonzero(flip)[:, 0], idx[flip]
        if len(w):
            q = f[:, n]
            r = q.sum(0)
            jx, jy = sum(EX[i] * q[i] for i in range(9)), sum(EY[i] * q[i] for i in range(9))
            sg = torch.where(ins[flip], 1.0, -1.0)
            Fx = sg * (jx - 0.5 * r * p["gx"] - r * self.X[w, 2])
            Fy = sg * (jy - 0.5 * r * p["gy"] - r * self.X[w, 3])
            G.index_add_(0, w, torch.stack([Fx, Fy, ax[flip] * Fy - ay[flip] * Fx], 1))
        if p["lj_psi"] and p["lj_rit"]:
            G += self.repulsion(y, x, ax, ay, ins)
        g = self.m * (self.rho_p - 1.0) / self.rho_p
        G[:, 0] += g * p["gx"]
        G[:, 1] += g * p["gy"]
        M = torch.stack([self.m, self.m, self.I], 1)
        V = self.X[:, 2:5]
        mid = torch.linalg.solve(torch.diag_embed(M) + 0.5 * Z, (M * V + 0.5 * G)[:, :, None])[:, :, 0]
        new = []
        for k, w, n, j, a in links:
            corr = 6.0 * WGT[k] * (mid[w] * a).sum(1)
            new.append((k, n, j, f[OPP[k]][j] + corr, f[k][n] - corr))
        for k, n, j, va, vb in new:
            f[k][n] = va
            f[OPP[k]][j] = vb
        self.prev = c
        X = self.X.clone()
        X[:, 0] += self.X[:, 2]
        X[:, 1] += self.X[:, 3]
        X[:, 5] += self.X[:, 4]
        X[:, 2:5] = 2.0 * mid - V
        if p["periodic_x"]:
            X[:, 0] %= self.nx
        if p["periodic_y"]:
            X[:, 1] %= self.ny
        self.X = X

    def step(self):
        p = self.p
        old = [None] * 9
        if any(self.any_bounce):
            old = [self.f[OPP[i]][:, self.bounce[i]] if self.any_bounce[i] else None for i in range(9)]
        if self.np:
            self.move_particles()
        f = self.f
        g = torch.empty_like(f)
        for i in range(9):
            g[i] = torch.roll(f[i], (EY[i], EX[i]), (1, 2))
            if old[i] is not None:
                g[i][:, self.bounce[i]] = old[i]
        f = g
        if p["inlet_outlet"]:
            c = f[:, :, 1:-1, 0]
            ru = p["rho_in"] - (c[0] + c[2] + c[4] + 2 * (c[3] + c[6] + c[7]))
            c[1] = c[3] + 2 / 3 * ru
            c[5] = c[7] - 0.5 * (c[2] - c[4]) + ru / 6
            c[8] = c[6] + 0.5 * (c[2] - c[4]) + ru / 6
            c = f[:, :, 1:-1, -1]
            ru = (c[0] + c[2] + c[4] + 2 * (c[1] + c[5] + c[8])) - p["rho_out"]
            c[3] = c[1] - 2 / 3 * ru
            c[7] = c[5] + 0.5 * (c[2] - c[4]) - ru / 6
            c[6] = c[8] - 0.5 * (c[2] - c[4]) - ru / 6
        rho, jx, jy = self.sums(f)
        if p["power_law"]:
            pxx = f[1] + f[3] + f[5] + f[6] + f[7] + f[8] - rho / 3 - jx * jx / rho
            pyy = f[2] + f[4] + f[5] + f[6] + f[7] + f[8] - rho / 3 - jy * jy / rho
            pxy = f[5] + f[7] - f[6] - f[8] - jx * jy / rho
            tau = self.local_tau(3.0 * torch.sqrt((pxy * pxy - pxx * pyy).abs()) / rho)
        else:
            tau = torch.full((), p["tau"], dtype=torch.float64, device=f.device)
        ux, uy = jx / rho + tau * p["gx"], jy / rho + tau * p["gy"]
        om, usq = 1.0 / tau, 1.5 * (ux * ux + uy * uy)
        for i in range(9):
            e = 3.0 * (EX[i] * ux + EY[i] * uy)
            f[i] -= om * (f[i] - WGT[i] * rho * (1.0 + e + 0.5 * e * e - usq))
        if bool((self.kT > 0).any()):
            th = _normals(self.node, self.t, self.dom, self.k0, self.k1)
            amp = torch.sqrt(3.0 * rho * self.kT * om * (2.0 - om))
            for i in range(9):
                f[i] += amp * sum(WGT[i] * _mode(k, i) * th[k - 3] for k in range(3, 9) if _mode(k, i))
        f[:, :, self.solid] = 0.0
        self.f = f
        self.t += 1

    def local_tau(self, A):
        """tau = 1/2 + 3 xi (A / tau)^(n-1), by bisection, clamped."""
        p, n = self.p, self.p["n_pl"]
        lo, hi = torch.full_like(A, p["tau_min"]), torch.full_like(A, p["tau_max"])
        c = 3.0 * p["xi_pl"] * A.clamp_min(1e-300) ** (n - 1.0)
        for _ in range(52):
            t = 0.5 * (lo + hi)
            low = t - 0.5 - c * t ** (1.0 - n) < 0
            lo, hi = torch.where(low, t, lo), torch.where(low, hi, t)
        return 0.5 * (lo + hi)

    @staticmethod
    def sums(f):
        return f.sum(0), f[1] + f[5] + f[8] - f[3] - f[6] - f[7], f[2] + f[5] + f[6] - f[4] - f[7] - f[8]

    def moments(self):
        rho, jx, jy = self.sums(self.f)
        safe = torch.where(self.solid, 1.0, rho)
        zero = torch.zeros_like(rho)
        return [rho] + [torch.where(self.solid, zero, (j - 0.5 * rho * g) / safe) for j, g in ((jx, self.p["gx"]), (jy, self.p["gy"]))]


def exact(case, seed):
    doms = _domains(case)
    out = {k: [None] * len(doms) for k in ("rho", "ux", "uy")}
    rec = [None] * len(doms)
    for size in sorted({(d[0], d[1]) for d in doms}):
        mine = [k for k, d in enumerate(doms) if (d[0], d[1]) == size]
        for at in range(0, len(mine), 16):  # several domains of a size at a time
            part = mine[at:at + 16]
            f = torch.stack([_populations(case, seed, k, *size, doms[k][2], doms[k][3]) for k in part], 1)
            e = _Exact(*size, [_seeded(doms[k][2], seed, k) for k in part], doms[part[0]][3], f, [doms[k][4] for k in part])
            states = []
            for _ in range(case["steps"]):
                e.step()
                if e.np:
                    states.append(e.X.clone())
            for key, v in zip(("rho", "ux", "uy"), e.moments()):
                for q, k in enumerate(part):
                    out[key][k] = v[q].reshape(-1)
            if e.np:
                states, first = torch.stack(states[-1:] + states[:-1]), 0  # the record of step t is at t mod steps
                for k in part:
                    rec[k] = states[:, first:first + len(doms[k][4])]
                    first += len(doms[k][4])
    got = {k: torch.cat(v) for k, v in out.items()}
    if any(len(d[4]) for d in doms):
        got["particles"] = torch.cat([r for r in rec if r is not None], 1).cpu()
    return got
