"""Measured workloads of the lattice Boltzmann library.

A case is one whole pass of a user's program through the public calls: an
initial state from density and velocity fields, a rollout of many updates, and
the observables (or the loss gradient) at its end.  The sizes are those of the
benchmark and the tests of this repository, with odd and ragged ones beside
them; ``draw`` spreads the same kinds of case over their whole ranges.

Kinds of case:
  box2d     D2Q9 on a periodic box or a force-driven channel with round
            obstacles: the parity and convergence studies of the 2D method
  cavity    D3Q19 BGK lid-driven cavity (halfway walls), the cavity with
            full-way walls and an equilibrium lid, or a periodic box
  sphere    D3Q27 KBC flow past a sphere, Zou-He inlet and outflow
  cylinder  D2Q9 Schafer-Turek cylinder: Bouzidi walls, regularized parabolic
            inflow, outflow, lift and drag read every few updates
  gradient  the kinetic-energy loss of a rollout and its gradient with respect
            to the initial fields, through torch.autograd
  batch     many independent small D2Q9 channels advanced together
  host      the cavity driven from page-locked host memory: mask and fields
            up, a rollout, observables down
"""
import math

import torch

from paper_2311_16080_gb300 import inputs as I
from paper_2311_16080_gb300 import xlb as X

FLUID, WALL, LID, INLET, OUTLET, EQ, FWALL = 0, 1, 2, 3, 4, 5, 6
DEV = "cuda" if torch.cuda.is_available() else "cpu"
LID_U = 0.05


def listed():
    return [
        # the Taylor-Green vortex of the accuracy study: the smallest lattice,
        # where the launch of each update costs more than its work
        dict(name="taylor_green_128_f32", kind="box2d", setup="periodic", nx=128, ny=128, storage="f32",
             collision="bgk", omega=1.25, steps=1000),
        # a small 2D channel of odd extent with obstacles and a body force, in
        # 16-bit storage
        dict(name="channel_203x67_f16", kind="box2d", setup="channel", nx=203, ny=67, storage="f16",
             collision="bgk", omega=1.25, steps=300),
        # the benchmark's lid-driven cavity
        dict(name="cavity_256_f32", kind="cavity", setup="cavity", nx=256, ny=256, nz=256, storage="f32",
             omega=1.85839, steps=40),
        # the same in the half-size storage a memory-limited user picks
        dict(name="cavity_256_f16", kind="cavity", setup="cavity", nx=256, ny=256, nz=256, storage="f16",
             omega=1.85839, steps=40),
        # a mid-size cavity of odd extents: rows are not a multiple of a warp
        dict(name="cavity_97x83x61_f32", kind="cavity", setup="cavity", nx=97, ny=83, nz=61, storage="f32",
             omega=1.7, steps=200),
        # odd extents in the stochastically rounded storage
        dict(name="cavity_161x130x127_bf16", kind="cavity", setup="cavity", nx=161, ny=130, nz=127, storage="bf16",
             omega=1.7, steps=50),
        # the KBC sphere channel at the benchmark's size: the largest state
        dict(name="sphere_512_f32", kind="sphere", nx=512, ny=256, nz=256, radius=32, storage="f32", omega=1.857,
             steps=10),
        # the same flow at half the resolution in 16-bit storage
        dict(name="sphere_256_f16", kind="sphere", nx=256, ny=128, nz=128, radius=16, storage="f16", omega=1.857,
             steps=20),
        # the cylinder benchmark at full resolution, graph replay, forces read
        dict(name="cylinder_80_f32", kind="cylinder", n_d=80, storage="f32", steps=400, every=100),
        # the differentiable rollout of the benchmark, checkpoints on the way
        dict(name="gradient_128_f32", kind="gradient", nx=128, ny=128, nz=128, storage="f32", omega=1.25, steps=100,
             every=20),
        # a batch of uneven channels, the autotuned launch
        dict(name="batch_1024_f32", kind="batch", domains=1024, geometry=1234, storage="f32", omega=1.25, steps=500),
        # one end-to-end call sequence on host buffers
        dict(name="host_cavity_160_f32", kind="host", nx=160, ny=160, nz=160, storage="f32", omega=1.8, steps=20),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["box2d", "box2d", "cavity", "cavity", "cavity", "sphere", "cylinder", "gradient", "batch",
                       "host"])
    storage = rng.choice(["f32", "f32", "f16", "bf16"])
    omega = round(rng.uniform(1.0, 1.85), 3)
    if kind == "box2d":
        nx, ny = _log_int(rng, 32, 600), _log_int(rng, 32, 600)
        steps = max(20, min(1000, _log_int(rng, 50, 1000), 60_000_000 // (nx * ny)))
        return dict(kind=kind, setup=rng.choice(["periodic", "channel"]), nx=nx, ny=ny, storage=storage,
                    collision=rng.choice(["bgk", "bgk", "kbc"]), omega=omega, steps=steps)
    if kind == "cavity":
        nx, ny, nz = (_log_int(rng, 24, 256) for _ in range(3))
        steps = max(5, min(_log_int(rng, 10, 200), 600_000_000 // (nx * ny * nz)))
        return dict(kind=kind, setup=rng.choice(["cavity", "cavity", "paper_cavity", "periodic"]), nx=nx, ny=ny,
                    nz=nz, storage=storage, omega=omega, steps=steps)
    if kind == "sphere":
        ny, nz = _log_int(rng, 32, 256), _log_int(rng, 32, 256)
        nx = _log_int(rng, 64, 512)
        steps = max(4, min(_log_int(rng, 5, 60), 300_000_000 // (nx * ny * nz)))
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, radius=max(3, min(ny, nz, nx // 2) // 8), storage=storage,
                    omega=round(rng.uniform(1.5, 1.857), 3), steps=steps)
    if kind == "cylinder":
        return dict(kind=kind, n_d=_log_int(rng, 10, 80), storage=rng.choice(["f32", "f32", "f16"]),
                    steps=rng.choice([100, 200, 300]), every=rng.choice([20, 50, 100]))
    if kind == "gradient":
        nx, ny, nz = (_log_int(rng, 20, 128) for _ in range(3))
        steps = _log_int(rng, 10, 100)
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, storage=rng.choice(["f32", "f32", "f16"]), omega=omega,
                    steps=steps, every=max(1, steps // rng.choice([1, 2, 5, 8])))
    if kind == "batch":
        return dict(kind=kind, domains=_log_int(rng, 32, 1024), geometry=rng.randrange(1 << 20), storage=storage,
                    omega=omega, steps=_log_int(rng, 20, 500))
    nx, ny, nz = (_log_int(rng, 32, 192) for _ in range(3))
    return dict(kind="host", nx=nx, ny=ny, nz=nz, storage=storage, omega=omega, steps=_log_int(rng, 5, 40))


# ---- set-ups -----------------------------------------------------------------

def _shape(case):
    return (case["ny"], case["nx"]) if case["kind"] == "box2d" else (case["nz"], case["ny"], case["nx"])


def _grid(shape):
    """Coordinates (x, y[, z]) as broadcastable arrays over a field's shape."""
    d = len(shape)
    out = []
    for a in range(d):
        view = [1] * d
        view[d - 1 - a] = -1
        out.append(torch.arange(shape[d - 1 - a], device=DEV).reshape(view))
    return out


def _mask(case):
    """Cell types of a case (uint8, x fastest), or None for a periodic box."""
    if case["kind"] == "box2d":
        if case["setup"] == "periodic":
            return None
        ny, nx = _shape(case)
        x, y = _grid((ny, nx))
        m = torch.zeros((ny, nx), dtype=torch.uint8, device=DEV)
        r = max(2, ny // 8)
        for cx, cy in ((nx // 4, ny // 2 + 1), (2 * nx // 3, ny // 3)):
            m[((x - cx) ** 2 + (y - cy) ** 2) <= r * r] = WALL
        m[0] = WALL
        m[-1] = WALL
        return m
    shape = _shape(case)
    m = torch.zeros(shape, dtype=torch.uint8, device=DEV)
    if case["kind"] == "sphere":
        x, y, z = _grid(shape)
        nz, ny, nx = shape
        m[(x - nx // 4) ** 2 + (y - ny // 2) ** 2 + (z - nz // 2) ** 2 <= case["radius"] ** 2] = WALL
        m[:, :, 0] = INLET
        m[:, :, -1] = OUTLET
        return m
    setup = case.get("setup", "cavity")
    if setup == "periodic" or case["kind"] == "gradient":
        return None
    wall, lid = (FWALL, EQ) if setup == "paper_cavity" else (WALL, LID)
    m[-1] = lid
    m[0] = wall
    m[:, 0] = wall
    m[:, -1] = wall
    m[:, :, 0] = wall
    m[:, :, -1] = wall
    return m


def _fields(shape, seed, u_mean=0.0, u_amp=0.03, rho_amp=2e-3):
    """A smooth seeded flow: long waves of random phase and direction, with
    some noise; rho around 1, u around u_mean along x."""
    g = torch.Generator(device="cpu").manual_seed(int(seed) + 77)
    gd = torch.Generator(device=DEV).manual_seed(int(seed) + 78)
    d = len(shape)
    xs = _grid(shape)
    out = []
    for a in range(d + 1):
        f = torch.zeros(shape, device=DEV)
        for _ in range(3):
            k = torch.randint(-2, 3, (d,), generator=g).tolist()
            ph = float(torch.rand((), generator=g)) * 2 * math.pi
            arg = ph
            for b in range(d):
                arg = arg + xs[b] * (2 * math.pi * k[b] / shape[d - 1 - b])
            f = f + torch.sin(arg) / 3
        f = f + 0.05 * torch.randn(shape, generator=gd, device=DEV)
        out.append(f)
    rho = (1.0 + rho_amp * out[0]).contiguous()
    u = u_amp * torch.stack(out[1:])
    u[0] += u_mean
    return rho, u.contiguous()


def _lattice_q(case):
    return {"box2d": 9, "cylinder": 9, "sphere": 27}.get(case["kind"], 19)


def _collision(case):
    return "kbc" if case["kind"] == "sphere" else case.get("collision", "bgk")


def _bc(case):
    """(type, rho, u) of the prescribed boundary of a case, or None."""
    if case["kind"] == "sphere":
        return INLET, 1.0, (0.04, 0.0, 0.0)
    if case["kind"] in ("cavity", "host"):
        return {"cavity": (LID, 1.0, (LID_U, 0.0, 0.0)), "paper_cavity": (EQ, 1.0, (LID_U, 0.0, 0.0))}.get(
            case.get("setup", "cavity"))
    return None


def _force(case):
    if case["kind"] == "box2d" and case["setup"] == "channel":
        nu = (1.0 / case["omega"] - 0.5) / 3.0
        return (8.0 * nu * 0.03 / (case["ny"] - 2) ** 2, 0.0, 0.0)
    return None


def _u_mean(case):
    return 0.04 if case["kind"] == "sphere" else 0.0


def _cylinder(case):
    """(mask, inflow field, links, q, omega, u) of the cylinder, numpy."""
    u = 0.03
    m, ctr, radius, uin = I.schafer_turek_2d(case["n_d"], u)
    cells, dirs, q = I.ball_links(m, ctr, radius, [list(v) for v in _C[9]])
    return m, uin, cells, dirs, q, 1.0 / (3.0 * u * case["n_d"] / 100.0 + 0.5), u


def _batch_domains(case):
    nu = (1.0 / case["omega"] - 0.5) / 3.0
    return I.batched_channels(case["domains"], seed=case["geometry"], nu=nu, u_max=0.05)


def _batch_fields(total, seed):
    g = torch.Generator(device=DEV).manual_seed(int(seed) + 79)
    rho = 1.0 + 2e-3 * torch.randn(total, generator=g, device=DEV)
    u = 0.01 * torch.randn((total, 2), generator=g, device=DEV)
    return rho, u.contiguous()


def _sync():
    if DEV == "cuda":
        torch.cuda.synchronize()


def prepare(case, seed):
    s = {"case": case, "stream": torch.cuda.Stream()}
    raw = s["stream"].cuda_stream
    kind = case["kind"]
    if kind == "batch":
        b = X.Batch(_batch_domains(case), case["omega"], case["storage"], stream=raw)
        total = sum(b.cells)
        s["rho0"], s["u0"] = _batch_fields(total, seed)
        s["rho"], s["u"] = torch.empty_like(s["rho0"]), torch.empty_like(s["u0"])
        _sync()
        b.set_masks()
        b.init(s["rho0"], s["u0"])
        b.step(1)
        b.tune(20)
        s["batch"] = b
        return s
    if kind == "cylinder":
        m, uin, cells, dirs, q, omega, u = _cylinder(case)
        sim = X.Simulation(9, (m.shape[1], m.shape[0]), omega, "bgk", case["storage"], stream=raw)
        rho, vel = _fields(m.shape, seed, u_amp=0.003)
        s["rho0"], s["u0"] = rho, (vel + torch.from_numpy(uin).to(DEV)).float().contiguous()
        _sync()
        sim.set_mask(m)
        sim.set_inlet_profile(uin.astype("float32"))
        sim.set_inlet_scheme("regularized")
        sim.set_wall_distances(cells, dirs, q.astype("float32"))
        sim.set_step_graph(case["every"])
        s["force"] = torch.zeros((case["steps"] // case["every"], 3), dtype=torch.float64, device=DEV)
        s["scale"] = 2.0 / (u * u * case["n_d"])
    else:
        shape = _shape(case)
        sim = X.Simulation(_lattice_q(case), tuple(reversed(shape)), case["omega"], _collision(case), case["storage"],
                           stream=raw)
        s["rho0"], s["u0"] = _fields(shape, seed, _u_mean(case))
        mask = _mask(case)
        _sync()
        if kind == "host":
            for k in ("rho0", "u0"):
                s[k] = s[k].cpu().pin_memory()
            s["mask"] = mask.cpu().pin_memory()
        elif mask is not None:
            sim.set_mask(mask)
        if kind != "host" and _bc(case):
            sim.set_bc(*_bc(case))
        if _force(case):
            sim.set_force(_force(case))
    s["sim"] = sim
    if kind == "gradient":
        s["rho0"].requires_grad_(True)
        s["u0"].requires_grad_(True)
        s["box"] = tuple(slice(3 * n // 8, max(3 * n // 8 + 1, 5 * n // 8)) for n in _shape(case))
    elif kind == "host":
        s["rho"], s["u"] = torch.empty_like(s["rho0"]).pin_memory(), torch.empty_like(s["u0"]).pin_memory()
    else:
        s["rho"], s["u"] = torch.empty_like(s["rho0"]), torch.empty_like(s["u0"])
    _sync()
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "batch":
        b = s["batch"]
        b.init(s["rho0"], s["u0"])
        b.step(case["steps"])
        X.xlb_batch_macroscopic(b.b, s["rho"], s["u"])
        return {"rho": s["rho"], "u": s["u"]}
    sim = s["sim"]
    if kind == "gradient":
        with torch.cuda.stream(s["stream"]):
            loss = X.rollout(sim, s["rho0"], case["steps"], case["every"], s["box"], u0=s["u0"])
            g_rho, g_u = torch.autograd.grad(loss, [s["rho0"], s["u0"]])
            return {"loss": loss.detach().float(), "grad_rho": g_rho, "grad_u": g_u}
    if kind == "host":
        sim.set_mask(s["mask"])
        sim.set_bc(*_bc(case))
    sim.init(s["rho0"], s["u0"])
    if kind == "cylinder":
        for k in range(case["steps"] // case["every"]):
            sim.step(case["every"])
            sim.wall_force(s["force"][k])
        sim.macroscopic(s["rho"], s["u"])
        # drag and lift coefficients of the cylinder (columns 0 and 1)
        return {"rho": s["rho"], "u": s["u"], "coefficients": (s["scale"] * s["force"][:, :2]).float()}
    sim.step(case["steps"])
    sim.macroscopic(s["rho"], s["u"])
    return {"rho": s["rho"], "u": s["u"]}


def _cells(case):
    if case["kind"] == "batch":
        return sum(d["nx"] * d["ny"] for d in _batch_domains(case))
    if case["kind"] == "cylinder":
        return (22 * case["n_d"] + 1) * (round(4.1 * case["n_d"]) + 2)
    n = 1
    for v in _shape(case):
        n *= v
    return n


def work(case):
    """Initial fields (and the host mask) read once, observables or gradients
    written once; additions and multiplications of the collisions."""
    n, q = _cells(case), _lattice_q(case) if case["kind"] != "batch" else 9
    d = 2 if q == 9 else 3
    per = {(9, "bgk"): 110, (9, "kbc"): 220, (19, "bgk"): 250, (27, "kbc"): 750}[(q, _collision(case))]
    updates = case["steps"]
    if case["kind"] == "gradient":
        per, updates = per + 420, case["steps"]
    by = 2 * (1 + d) * 4 * n + (n if case["kind"] == "host" else 0)
    return {"bytes": by, "flops": per * n * updates}


# ---- the same in 64 bits, plain torch -------------------------------------------

_C = {9: [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (1, -1), (-1, 1), (-1, -1)],
      19: [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (-1, 0, 0), (0, -1, 0), (0, 0, -1), (1, 1, 0), (1, -1, 0),
           (-1, 1, 0), (-1, -1, 0), (1, 0, 1), (1, 0, -1), (-1, 0, 1), (-1, 0, -1), (0, 1, 1), (0, 1, -1),
           (0, -1, 1), (0, -1, -1)]}
_C[27] = _C[19] + [(a, b, c) for a in (1, -1) for b in (1, -1) for c in (1, -1)]
_W = {9: (4 / 9, 1 / 9, 1 / 36), 19: (1 / 3, 1 / 18, 1 / 36), 27: (8 / 27, 2 / 27, 1 / 54, 1 / 216)}


class _Exact:
    """Flat FP64 lattice: populations f[i, cell]; streaming is one gather by a
    table of source slots, which carries the boundary rules."""

    def __init__(self, q, omega, collision, force=None):
        self.q, self.omega, self.coll, self.force = q, float(omega), collision, force
        self.c = _C[q]
        self.d = len(self.c[0])
        self.w = [_W[q][sum(v * v for v in ci)] for ci in self.c]
        self.opp = [self.c.index(tuple(-v for v in ci)) for ci in self.c]

    def dot(self, i, u):
        s = 0.0
        for a, ca in enumerate(self.c[i]):
            if ca:
                s = s + ca * u[a]
        return s

    def eq(self, i, rho, u, usq):
        cu = self.dot(i, u)
        return self.w[i] * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * usq)

    def moments(self, f):
        rho = f[0]
        for i in range(1, self.q):
            rho = rho + f[i]
        j = []
        for a in range(self.d):
            s = 0.0
            for i in range(self.q):
                if self.c[i][a]:
                    s = s + self.c[i][a] * f[i]
            j.append(s)
        return rho, j

    def table(self, types, shape):
        """Source slots of the pull and its constant terms, from the mask."""
        n = types.numel()
        shape3 = shape if self.d == 3 else (1,) + tuple(shape)
        nz, ny, nx = shape3
        cell = torch.arange(n, device=DEV)
        x, y, z = cell % nx, cell // nx % ny, cell // (nx * ny)
        idx = torch.empty((self.q, n), dtype=torch.int64, device=DEV)
        add = {}
        for i, ci in enumerate(self.c):
            cz = ci[2] if self.d == 3 else 0
            src = (((z - cz) % nz) * ny + (y - ci[1]) % ny) * nx + (x - ci[0]) % nx
            t = types[src]
            idx[i] = torch.where((t == WALL) | (t == LID), self.opp[i] * n + cell, i * n + src)
            if (t == LID).any():
                cu = sum(a * b for a, b in zip(ci, self.lid[1]))
                add[i] = (t == LID).double() * (6.0 * self.w[i] * self.lid[0] * cu)
            if (t == EQ).any():
                add.setdefault(i, torch.zeros(n, dtype=torch.float64, device=DEV))
                u = [float(v) for v in self.eqv[1]]
                add[i] = torch.where(t == EQ, self.eq(i, self.eqv[0], u, sum(v * v for v in u)), add[i])
                self.zero[i] = t == EQ
        out = torch.nonzero(types == OUTLET).reshape(-1)
        for i, ci in enumerate(self.c):
            if ci[0] == -1 and out.numel():
                idx[i, out] = idx[i, out - 1]
        self.idx, self.add, self.n = idx, add, n
        self.types, self.x_shape = types, shape3

    lid, eqv = (1.0, (0.0, 0.0, 0.0)), (1.0, (0.0, 0.0, 0.0))
    inlet = None  # (cells, velocity [d][cells], regularized)
    links = None  # (slot, slot a, weight a, slot b, weight b)

    def prepare(self, types, shape):
        self.zero = {}
        self.table(types, shape)
        self.solid = ~((types == FLUID) | (types == INLET) | (types == OUTLET))
        self.fwall = torch.nonzero(types == FWALL).reshape(-1)

    def init(self, rho, u):
        usq = sum(v * v for v in u)
        f = torch.stack([self.eq(i, rho, u, usq) for i in range(self.q)])
        if self.fwall.numel():
            f[:, self.fwall] = torch.tensor(self.w, dtype=torch.float64, device=DEV)[:, None]
        return f

    def collide(self, f):
        rho, j = self.moments(f)
        u = [v / rho for v in j]
        usq = sum(v * v for v in u)
        if self.coll == "bgk":
            h = [f[i] + self.omega * (self.eq(i, rho, u, usq) - f[i]) for i in range(self.q)]
        else:
            h = self.kbc(f, rho, u, usq)
        if self.force is not None:
            v = [u[a] + self.force[a] / rho for a in range(self.d)]
            vsq = sum(x * x for x in v)
            h = [h[i] + self.eq(i, rho, v, vsq) - self.eq(i, rho, u, usq) for i in range(self.q)]
        h = torch.stack(h)
        if self.fwall.numel():
            h[:, self.fwall] = f[self.opp][:, self.fwall]
        return h

    def kbc(self, f, rho, u, usq):
        d, q = self.d, self.q
        g = [f[i] - self.eq(i, rho, u, usq) for i in range(q)]
        P = {}
        for a in range(d):
            for b in range(a, d):
                P[a, b] = sum(self.c[i][a] * self.c[i][b] * g[i] for i in range(q) if self.c[i][a] * self.c[i][b])
        tr = sum(P[a, a] for a in range(d)) / d
        s = []
        for ci in self.c:
            nz = [a for a in range(d) if ci[a]]
            s.append(0.5 * (P[nz[0], nz[0]] - tr) if len(nz) == 1 else
                     0.25 * ci[nz[0]] * ci[nz[1]] * P[nz[0], nz[1]] if len(nz) == 2 else 0.0)
        beta = 0.5 * self.omega
        sh = hh = 0.0
        for i in range(q):
            e = self.eq(i, rho, u, usq)
            h = g[i] - s[i]
            sh, hh = sh + s[i] * h / e, hh + h * h / e
        tiny = hh < 1e-30
        gamma = 1 / beta - (2 - 1 / beta) * sh / torch.where(tiny, torch.ones_like(hh), hh)
        gamma = torch.where(tiny, torch.full_like(hh, 2.0), gamma)
        return [f[i] - beta * (2 * s[i] + gamma * (g[i] - s[i])) for i in range(q)]

    def stream(self, h):
        flat = h.reshape(-1)
        f = torch.gather(flat, 0, self.idx.reshape(-1)).reshape(self.q, self.n)
        for i, t in self.add.items():
            if i in self.zero:
                f[i] = torch.where(self.zero[i], t, f[i] + t)
            else:
                f[i] = f[i] + t
        if self.links is not None:
            slot, a, wa, b, wb = self.links
            f.view(-1)[slot] = wa * flat[a] + wb * flat[b]
        if self.inlet is not None:
            self.inlet_rule(f)
        return f

    def inlet_rule(self, f):
        cells, u, regularized = self.inlet
        g = [f[i, cells] for i in range(self.q)]
        rho = sum(g[i] * (1 if self.c[i][0] == 0 else 2) for i in range(self.q) if self.c[i][0] <= 0) / (1.0 - u[0])
        usq = sum(v * v for v in u)
        e = [self.eq(i, rho, u, usq) for i in range(self.q)]
        k = [g[self.opp[i]] - e[self.opp[i]] if self.c[i][0] == 1 else g[i] - e[i] for i in range(self.q)]
        if regularized:
            d = self.d
            P = [[sum(self.c[i][a] * self.c[i][b] * k[i] for i in range(self.q)) for b in range(d)] for a in range(d)]
            k = [4.5 * self.w[i] * sum((self.c[i][a] * self.c[i][b] - (a == b) / 3.0) * P[a][b]
                                       for a in range(d) for b in range(d)) for i in range(self.q)]
        for i in range(self.q):
            if regularized or self.c[i][0] == 1:
                f[i, cells] = e[i] + k[i]

    def observables(self, f):
        rho, j = self.moments(f)
        F = self.force if self.force is not None else [0.0] * self.d
        u = torch.stack([(j[a] + 0.5 * F[a]) / rho for a in range(self.d)])
        rho = torch.where(self.solid, torch.zeros_like(rho), rho)
        u = torch.where(self.solid, torch.zeros_like(u), u)
        e = self.types == EQ
        if e.any():
            rho = torch.where(e, torch.full_like(rho, self.eqv[0]), rho)
            ev = torch.tensor(self.eqv[1][:self.d], dtype=torch.float64, device=DEV)[:, None]
            u = torch.where(e, ev, u)
        return rho, u


def _f32(v):
    """The value a float32 argument of the library holds."""
    return [float(torch.tensor(x, dtype=torch.float32)) for x in v]


def _exact_gradient(case, seed):
    shape = _shape(case)
    ex = _Exact(19, case["omega"], "bgk")
    types = torch.zeros(shape, dtype=torch.uint8, device=DEV).reshape(-1)
    ex.prepare(types, shape)
    r32, u32 = _fields(shape, seed)
    rho0 = r32.double().reshape(-1).requires_grad_(True)
    u0 = u32.double().reshape(3, -1).requires_grad_(True)
    states = [ex.init(rho0, [u0[a] for a in range(3)]).detach()]
    for _ in range(case["steps"]):
        states.append(ex.stream(ex.collide(states[-1])))
    box = torch.zeros(shape, dtype=torch.float64, device=DEV)
    box[tuple(slice(3 * n // 8, max(3 * n // 8 + 1, 5 * n // 8)) for n in shape)] = 1.0
    f = states.pop().requires_grad_(True)
    rho, u = ex.observables(f)
    loss = (0.5 * box.reshape(-1) * rho * (u * u).sum(0)).sum()
    (g,) = torch.autograd.grad(loss, [f])
    while states:
        f = states.pop().requires_grad_(True)
        (g,) = torch.autograd.grad(ex.stream(ex.collide(f)), [f], g)
    gr, gu = torch.autograd.grad(ex.init(rho0, [u0[a] for a in range(3)]), [rho0, u0], g)
    return {"loss": loss.detach(), "grad_rho": gr.reshape(shape), "grad_u": gu.reshape((3,) + shape)}


def _exact_cylinder(case, seed):
    m, uin, cells, dirs, q, omega, u_mean = _cylinder(case)
    shape = m.shape
    types = torch.from_numpy(m).to(DEV).reshape(-1)
    ex = _Exact(9, omega, "bgk")
    ex.prepare(types, shape)
    n, nx = ex.n, shape[1]
    inl = torch.nonzero(types == INLET).reshape(-1)
    prof = torch.from_numpy(uin.astype("float32")).to(DEV).double().reshape(2, -1)
    ex.inlet = (inl, [prof[a][inl] for a in range(2)], True)
    slot, sa, wa, sb, wb, force = [], [], [], [], [], []
    fluid = (types == FLUID).cpu()
    for x, i, qq in zip(cells.tolist(), dirs.tolist(), q.astype("float32").tolist()):
        j = ex.opp[i]
        back = x + ex.c[j][0] + nx * ex.c[j][1]
        slot.append(j * n + x)
        sa.append(i * n + x)
        force.append((x, i))
        if qq >= 0.5:
            wa.append(0.5 / qq), sb.append(j * n + x), wb.append(1.0 - 0.5 / qq)
        elif fluid[back]:
            wa.append(2 * qq), sb.append(i * n + back), wb.append(1.0 - 2 * qq)
        else:
            wa.append(1.0), sb.append(i * n + x), wb.append(0.0)
    t = lambda v, k: torch.tensor(v, dtype=k, device=DEV)  # noqa: E731
    ex.links = (t(slot, torch.int64), t(sa, torch.int64), t(wa, torch.float64), t(sb, torch.int64),
                t(wb, torch.float64))
    cvec = t([[float(v) for v in ex.c[i]] for _, i in force], torch.float64)
    rho, vel = _fields(shape, seed, u_amp=0.003)
    u0 = (vel + torch.from_numpy(uin).to(DEV)).float().double().reshape(2, -1)
    f = ex.init(rho.double().reshape(-1), [u0[a] for a in range(2)])
    co = []
    for k in range(case["steps"]):
        h = ex.collide(f)
        f = ex.stream(h)
        if (k + 1) % case["every"] == 0:
            v = h.reshape(-1)[ex.links[1]] + f.reshape(-1)[ex.links[0]]
            co.append((cvec * v[:, None]).sum(0) * (2.0 / (u_mean * u_mean * case["n_d"])))
    rho, u = ex.observables(f)
    return {"rho": rho.reshape(shape), "u": u.reshape((2,) + tuple(shape)), "coefficients": torch.stack(co)}


def _exact_batch(case, seed):
    doms = _batch_domains(case)
    ex = _Exact(9, case["omega"], "bgk")
    n = sum(d["nx"] * d["ny"] for d in doms)
    idx = torch.empty((9, n), dtype=torch.int64, device=DEV)
    types = torch.empty(n, dtype=torch.uint8, device=DEV)
    F = torch.empty((2, n), dtype=torch.float64, device=DEV)
    o = 0
    for dom in doms:
        k = dom["nx"] * dom["ny"]
        one = _Exact(9, 1.0, "bgk")
        types[o:o + k] = torch.from_numpy(dom["mask"]).to(DEV).reshape(-1)
        one.zero = {}
        one.table(types[o:o + k], (dom["ny"], dom["nx"]))
        idx[:, o:o + k] = one.idx // k * n + one.idx % k + o
        F[:, o:o + k] = torch.tensor(_f32(dom["force"]), dtype=torch.float64, device=DEV)[:, None]
        o += k
    ex.idx, ex.add, ex.zero, ex.n, ex.types = idx, {}, {}, n, types
    ex.solid, ex.fwall, ex.force = types != FLUID, torch.zeros(0, dtype=torch.int64), F
    rho, u = _batch_fields(n, seed)
    f = ex.init(rho.double(), [u[:, a].double() for a in range(2)])
    for _ in range(case["steps"]):
        f = ex.stream(ex.collide(f))
    rho, u = ex.observables(f)
    return {"rho": rho, "u": u.t().contiguous()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "gradient":
        return _exact_gradient(case, seed)
    if kind == "cylinder":
        return _exact_cylinder(case, seed)
    if kind == "batch":
        return _exact_batch(case, seed)
    shape = _shape(case)
    mask = _mask(case)
    types = (mask if mask is not None else torch.zeros(shape, dtype=torch.uint8, device=DEV)).reshape(-1)
    ex = _Exact(_lattice_q(case), case["omega"], _collision(case), _f32(_force(case)) if _force(case) else None)
    bc = _bc(case)
    if bc:
        v = (bc[1], tuple(_f32(bc[2])))
        ex.lid = v if bc[0] == LID else ex.lid
        ex.eqv = v if bc[0] == EQ else ex.eqv
    ex.prepare(types, shape)
    if bc and bc[0] == INLET:
        cells = torch.nonzero(types == INLET).reshape(-1)
        ex.inlet = (cells, _f32(bc[2]), False)
    rho, u = _fields(shape, seed, _u_mean(case))
    d = len(shape)
    f = ex.init(rho.double().reshape(-1), [u[a].double().reshape(-1) for a in range(d)])
    for _ in range(case["steps"]):
        f = ex.stream(ex.collide(f))
    rho, u = ex.observables(f)
    return {"rho": rho.reshape(shape), "u": u.reshape((d,) + tuple(shape))}
