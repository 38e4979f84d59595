"""The performance cases of the library: what a user's program has it do.

A case is a domain (or a batch of domains) with one of the paper's set-ups,
advanced by Domain.step(n) or Batch.step(n), or read by Domain.observables().
The domains are created as a host program with its own device memory creates
them (the allocator callbacks of lbmp_create_ex), so the outputs of a pass are
the library's own device arrays: both current population sets, whole, in the
native layout (FP32 [a][cell]; 16-bit storage: one FP32 reference per cell and
the codes [a without the rest][cell]), and the stored phi u of the reduced
phase lattice.

exact() is the same update in plain torch at 64 bits, from the formulas of
arXiv 2101.06769, Sec. 2.2 and 2.3, with none of the library's code.
"""
import math

import numpy as np
import torch

from paper_2101_06769_gb300 import FLAG_PHASE_REDUCED, Batch, Domain
from paper_2101_06769_gb300.lbmp import FLAG_AA, make_allocator

FP32, FP16, BF16 = 0, 1, 2
CODE_TYPE = {FP16: torch.float16, BF16: torch.bfloat16}
CODE_SCALE = {FP16: 2.0 ** 20, BF16: 1.0}


# ------------------------------------------------------------------ the cases
def case(name, kind, nx, ny, nz, steps, storage=FP32, form="full", walls=True, stream=False, ratio=3.0):
    """kind: "rt" (Rayleigh-Taylor), "splash" (drop on a sheet), "drop"
    (static drop), "half" (the 2-D impact's half domain with a symmetry x
    axis), "mix" (a batch) or "observe" (the FP64 observables of an RT
    domain); nz = 1 selects D2Q9.  form: "full", "reduced" (D3Q7 / D2Q5 phase
    field) or "aa" (in-place storage); ratio: density ratio."""
    return dict(name=name, kind=kind, nx=nx, ny=ny, nz=nz, steps=steps, storage=storage, form=form, walls=walls,
                stream=stream, ratio=ratio)


def listed():
    return [
        # the 2-D Rayleigh-Taylor workload (the shipped rt2d case): the smallest domain
        # that is run in earnest, where launches and latency count; a caller's own
        # stream, and a step count that is no multiple of the graph's
        case("rt2d_64x256", "rt", 64, 256, 1, 37, stream=True),
        # the paper's 2-D droplet impact (the shipped splash2d_k56 case): half domain with
        # a symmetry axis, density ratio 1000, an odd step count on the default stream
        case("splash2d_400x250", "half", 400, 250, 1, 21, ratio=1000.0),
        # a 2-D domain large enough for HBM to count (the D2Q9 throughput size)
        case("rt2d_4096x2048", "rt", 4096, 2048, 1, 4),
        # 2-D in 16-bit storage at a ragged (even) width
        case("rt2d_bf16_1350x1021", "rt", 1350, 1021, 1, 8, storage=BF16),
        # the smallest 3-D size of the serving stream, alone
        case("rt3d_64", "rt", 64, 64, 64, 21, stream=True),
        # odd, ragged sizes: a periodic 3-D drop at density ratio 20
        case("drop3d_141x107x93", "drop", 141, 107, 93, 7, walls=False, ratio=20.0),
        # the benchmark workload: 3-D Rayleigh-Taylor, FP32
        case("rt3d_128x128x512", "rt", 128, 128, 512, 4),
        # the same in 16-bit storage (half the state: what makes the largest splash fit)
        case("rt3d_fp16_128x128x512", "rt", 128, 128, 512, 4, storage=FP16),
        # the same with the D3Q7 phase field, the cheapest FP32 form of the update
        case("rt3d_reduced_128x128x512", "rt", 128, 128, 512, 4, form="reduced"),
        # the 3-D droplet impact (the shipped splash3d case): density ratio 1000, the
        # largest domain here
        case("splash3d_384x384x192", "splash", 384, 384, 192, 2, ratio=1000.0),
        # continuous batching: 2-D and 3-D requests of uneven sizes advanced together
        case("batch_mix", "mix", 128, 128, 128, 16, stream=True),
        # the observables that the serving loop and a monitored run read between rounds
        case("observables_128x128x512", "observe", 128, 128, 512, 1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rt2", "rt2", "half", "bf2", "rt3", "rt3", "drop3", "st3", "red3", "splash", "aa3", "mix",
                       "observe"])
    stream = rng.random() < 0.5
    if kind in ("rt2", "half", "bf2"):
        nx, ny = _log(rng, 48, 3000), _log(rng, 64, 2000)
        n = max(2, min(40, int(2e7 / (nx * ny)) + rng.randint(0, 1)))
        if kind == "half":
            return case("", "half", nx, max(128, ny), 1, n, stream=stream, ratio=1000.0,
                        form=rng.choice(["full", "reduced"]))
        if kind == "bf2":
            return case("", "rt", nx + nx % 2, ny, 1, n, storage=rng.choice([FP16, BF16]), stream=stream)
        return case("", "rt", nx, ny, 1, n, form=rng.choice(["full", "full", "reduced"]), stream=stream,
                    ratio=rng.choice([3.0, 9.0]))
    nx, ny, nz = _log(rng, 32, 240), _log(rng, 32, 240), _log(rng, 32, 300)
    n = max(2, min(24, int(2e7 / (nx * ny * nz)) + rng.randint(0, 1)))
    if kind == "drop3":
        return case("", "drop", nx, ny, nz, n, walls=False, stream=stream, ratio=20.0)
    if kind == "st3":
        return case("", "rt", nx + nx % 2, ny, nz, n, storage=rng.choice([FP16, BF16]), stream=stream)
    if kind == "red3":
        return case("", "rt", nx, ny, nz, n, form="reduced", stream=stream)
    if kind == "splash":
        return case("", "splash", nx, ny, max(64, nz), n, stream=stream, ratio=1000.0)
    if kind == "aa3":
        return case("", "rt", nx, ny, nz, n + n % 2, form="aa", stream=stream)
    if kind == "mix":
        s = 32 * rng.randint(2, 4)
        return case("", "mix", s, s, s, rng.randint(3, 20), stream=True)
    if kind == "observe":
        return case("", "observe", nx, ny, nz, 1, storage=rng.choice([FP32, FP32, FP16]) if nx % 2 == 0 else FP32)
    return case("", "rt", nx, ny, nz, n, stream=stream, ratio=rng.choice([3.0, 9.0]))


# ------------------------------------------------- the set-ups (both sides use them)
def setup(c, seed):
    """Lattice, grid, boundaries, parameters and initial condition of a case:
    the paper's set-ups as the shipped case files and the serving stream scale
    them.  The interface amplitude or the drop's size varies with the seed, as
    does the velocity noise."""
    D = 2 if c["nz"] == 1 else 3
    dims = (c["nx"], c["ny"], c["nz"])
    nv = dims[D - 1]
    vary = 1.0 + 0.1 * ((seed * 2654435761) % 1000) / 1000.0
    vert = 0 if c["walls"] else 1
    periodic = (1, 1, vert) if D == 3 else (1, vert, 1)
    side = float(dims[0])
    if c["kind"] in ("rt", "observe"):
        phys = dict(rho_ratio=c["ratio"], nu_ratio=1.0, Re=256.0 if D == 2 else 1024.0, g_accel=0.04 ** 2 / side,
                    L_ref=side, mobility=0.02, width=5.0)
        init = ("rt", [nv / 2.0, 0.05 * side * vary, 1e-2, 1.0])
    elif c["kind"] == "splash":
        dd = max(16.0, min(dims[0], nv) / 3.0) * vary
        phys = dict(rho_ratio=c["ratio"], nu_ratio=15.0, We=8000.0, Re=1000.0, U0=0.05, L_ref=dd, mobility=0.1,
                    width=4.0)
        init = ("drop_sheet", [dd, 0.2 * dd, 0.05, 1e-4])
    elif c["kind"] == "half":
        periodic = (2, 0, 1)
        dd = 0.4 * nv * vary
        phys = dict(rho_ratio=c["ratio"], nu_ratio=15.0, We=220.0, Re=200.0, U0=0.05, L_ref=dd, mobility=0.1,
                    width=5.0)
        init = ("drop_sheet", [dd, 0.2 * dd, 0.05, 1e-4, -0.5])
    else:
        r = 0.25 * min(dims[:D]) * vary
        phys = dict(rho_ratio=c["ratio"], nu_ratio=2.0, nu_h=0.05, sigma=1e-2, mobility=0.02, width=4.0, U0=0.01,
                    L_ref=r)
        init = ("drop_static", [r, 1.0, 1e-2])
    phys["storage"] = c["storage"]
    phys["flags"] = {"full": 0, "reduced": FLAG_PHASE_REDUCED, "aa": FLAG_AA}[c["form"]]
    return D, dims, periodic, phys, init, 1 + seed % 1000003


def members(c):
    """The requests of a batch case, as cases of their own: uneven 3-D and 2-D
    sizes around the given side, of both set-ups of the serving stream."""
    s = c["nx"]
    return [case("", "rt", s, s, s, 1), case("", "splash", s // 2, s // 2, s, 1, ratio=100.0),
            case("", "rt", s // 2, s // 2, s // 2, 1, ratio=9.0), case("", "rt", 3 * s // 4, s // 2 + 1, s, 1),
            case("", "rt", 2 * s, 2 * s, 1, 1), case("", "rt", s, 4 * s, 1, 1, ratio=9.0),
            case("", "half", 3 * s, 2 * s, 1, 1, ratio=1000.0), case("", "rt", s // 2, s, 1, 1)]


# ---------------------------------------------------------------- prepare and run
class Held:
    """Device memory of one domain, as a program that owns it hands it out:
    the arrays in the order the library asks for them (f' and g of the first
    set, f' and g of the second, ...)."""

    def __init__(self):
        self.order, self.place = [], {}
        self.allocator = make_allocator(self.take, self.give)

    def take(self, nbytes, stream):
        t = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        self.place[t.data_ptr()] = len(self.order)
        self.order.append(t)
        return t.data_ptr()

    def give(self, ptr, nbytes, stream):
        self.order[self.place.pop(ptr)] = None


def make_domain(c, seed, stream):
    D, dims, periodic, phys, (name, args), s = setup(c, seed)
    held = Held()
    d = Domain(D, dims, periodic, stream=stream, allocator=held.allocator, **phys)
    d.init(name, args, seed=s)
    return dict(case=c, domain=d, held=held, taken=0)


def prepare(c, seed):
    # the stream outlives the domains that use it
    stream = torch.cuda.Stream() if c["stream"] else None
    handle = stream.cuda_stream if stream is not None else None
    if c["kind"] != "mix":
        return dict(stream=stream, **make_domain(c, seed, handle))
    b = Batch(stream=handle)
    doms = [make_domain(m, seed + k, handle) for k, m in enumerate(members(c))]
    for m in doms:
        b.add(m["domain"], 1 << 30)
    return dict(stream=stream, case=c, batch=b, domains=doms)


def current(m):
    """The current population sets of a domain: its own device arrays."""
    c, bufs = m["case"], m["held"].order
    D = 2 if c["nz"] == 1 else 3
    n = c["nx"] * c["ny"] * c["nz"]
    k = 0 if c["form"] == "aa" else m["taken"] & 1
    out = {}
    for name, b in (("f", bufs[2 * k]), ("g", bufs[2 * k + 1])):
        if c["storage"] == FP32:
            out[name] = b.view(torch.float32)
        else:
            out[name + "_ref"] = b[:4 * n].view(torch.float32)
            out[name + "_codes"] = b[4 * n:].view(CODE_TYPE[c["storage"]])
    if c["form"] == "reduced":
        out["phi_u"] = bufs[4][:4 * D * n].view(torch.float32)
    return out


def run(state):
    c = state["case"]
    if c["kind"] == "mix":
        state["batch"].step(c["steps"])
        for m in state["domains"]:
            m["taken"] += c["steps"]
        return [current(m) for m in state["domains"]]
    if c["kind"] == "observe":
        return state["domain"].observables().as_dict()
    state["domain"].step(c["steps"])
    state["taken"] += c["steps"]
    return current(state)


def work(c):
    """Every population is read once and written once per step (with the
    stored phi u of the reduced phase lattice); the observables read the
    current sets once.  The operations are those of one cell update, counted
    from the formulas."""
    if c["kind"] == "mix":
        w = [work(dict(m, steps=c["steps"])) for m in members(c)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    D = 2 if c["nz"] == 1 else 3
    q = 9 if D == 2 else 27
    cells = c["nx"] * c["ny"] * c["nz"]
    each = 4.0 * q if c["storage"] == FP32 else 4.0 + 2.0 * (q - 1)
    both = each + (4.0 * (2 * D + 1 + D) if c["form"] == "reduced" else each)
    if c["kind"] == "observe":
        return {"bytes": both * cells, "flops": (400.0 if D == 3 else 150.0) * cells}
    return {"bytes": 2.0 * both * cells * c["steps"], "flops": (1900.0 if D == 3 else 600.0) * cells * c["steps"]}


# ------------------------------------------------------------------------- exact
def _dirs(D):
    return [(x, y, z) for z in ((-1, 0, 1) if D == 3 else (0,)) for y in (-1, 0, 1) for x in (-1, 0, 1)]


def _w1(c):
    return 2.0 / 3.0 if c == 0 else 1.0 / 6.0


class Exact:
    """The coupled update of one domain in 64 bits; arrays are [z][y][x]."""

    def __init__(self, c, seed):
        self.c = c
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.D, dims, self.periodic, p, (self.case, self.args), self.seed = setup(c, seed)
        D = self.D
        self.nx, self.ny, self.nz = dims
        self.sym = self.periodic[0] == 2
        self.wall = self.periodic[D - 1] == 0
        self.reduced = c["form"] == "reduced"
        self.C = _dirs(D)
        self.Q = len(self.C)
        self.W = [_w1(x) * _w1(y) * (_w1(z) if D == 3 else 1.0) for x, y, z in self.C]
        self.index = {d: a for a, d in enumerate(self.C)}
        # phase lattice: directions, weights, 1/cs2
        if self.reduced:
            self.G = [d for d in self.C if sum(abs(v) for v in d) <= 1]
            rest, face = (0.25, 0.125) if D == 3 else (1 / 3, 1 / 6)
            self.GW = [rest if d == (0, 0, 0) else face for d in self.G]
            self.ics2g = 4.0 if D == 3 else 3.0
        else:
            self.G, self.GW, self.ics2g = self.C, self.W, 3.0
        # parameters (heavy density 1)
        self.rho_l = 1.0 / p["rho_ratio"]
        self.width, self.g_accel = p["width"], p.get("g_accel", 0.0)
        self.U = p.get("U0") or math.sqrt(self.g_accel * p["L_ref"])
        self.nu_h = p.get("nu_h") or self.U * p["L_ref"] / p["Re"]
        self.nu_l = self.nu_h * p["nu_ratio"]
        self.sigma = p["sigma"] if "sigma" in p else (p["L_ref"] * self.U ** 2 / p["We"] if "We" in p else 0.0)
        self.beta, self.kappa = 12 * self.sigma / self.width, 1.5 * self.sigma * self.width
        self.tau = p["mobility"] * self.ics2g + 0.5
        self.lam = 1 - 0.5 / self.tau

    def coords(self):
        def ar(n):
            return torch.arange(n, dtype=torch.float64, device=self.dev)
        return ar(self.nx).view(1, 1, -1), ar(self.ny).view(1, -1, 1), ar(self.nz).view(-1, 1, 1)

    def noise(self, k):
        """Uniform numbers in [-1, 1) of splitmix64(seed, 3 cell + k)."""
        def shr(v, s):
            return (v >> s) & ((1 << (64 - s)) - 1)

        def wrap(v):
            v &= (1 << 64) - 1
            return v - (1 << 64) if v >= 1 << 63 else v
        i = torch.arange(self.nx * self.ny * self.nz, dtype=torch.int64, device=self.dev)
        z = (3 * i + (k + 1)) * wrap(0x9E3779B97F4A7C15) + self.seed
        z = (z ^ shr(z, 30)) * wrap(0xBF58476D1CE4E5B9)
        z = (z ^ shr(z, 27)) * wrap(0x94D049BB133111EB)
        z = z ^ shr(z, 31)
        return (2.0 * shr(z, 11).double() / 2.0 ** 53 - 1.0).view(self.nz, self.ny, self.nx)

    def start(self):
        """The initial populations, rounded to the 32 bits they are stored in."""
        D, a, W = self.D, self.args, self.width
        X = self.coords()
        n = (self.nx, self.ny, self.nz)
        v = D - 1
        zero = torch.zeros(self.nz, self.ny, self.nx, dtype=torch.float64, device=self.dev)

        def prof(d):
            return 0.5 * (1 + torch.tanh(2 * d / W))
        u = [zero, zero, zero]
        pr = zero
        if self.case == "rt":
            h = a[0] + a[1] * torch.cos(2 * math.pi * X[0] / self.nx)
            if D == 3:
                h = h + a[1] * torch.cos(2 * math.pi * X[1] / self.ny)
            phi = prof(X[v] - h) + zero
            t = (2 * (X[v] - h) / W).abs() + zero
            pr = -self.g_accel * (1 - self.rho_l) * 0.25 * W * (t + torch.log1p(torch.exp(-2 * t)) - math.log(2.0))
            amp = a[2]
        elif self.case == "drop_static":
            r = torch.sqrt(sum((X[k] - n[k] // 2) ** 2 for k in range(D)))
            phi = prof(a[0] - r) + zero
            pr = (2.0 if D == 3 else 1.0) * self.sigma / a[0] * phi
            amp = a[2]
        else:
            centre = [a[4] if len(a) > 4 else n[k] // 2 for k in range(D)]
            centre[v] = a[1] + 0.5 * a[0] + 2 * W
            d = 0.5 * a[0] - torch.sqrt(sum((X[k] - centre[k]) ** 2 for k in range(D)))
            phi = prof(torch.maximum(d, a[1] - X[v])) + zero
            u[v] = -a[2] * prof(d) + zero
            amp = a[3]
        for k in range(D):
            u[k] = u[k] + amp * self.U * self.noise(k) * phi
        rho = self.rho_l + (1 - self.rho_l) * phi
        uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        f = [self.W[i] * pr + rho / 3 * self.gdev(i, u, uu) for i in range(self.Q)]
        if self.reduced:
            g = [w * phi * (1 + self.ics2g * self.dot(d, u)) for d, w in zip(self.G, self.GW)]
        else:
            g = [phi * (self.W[i] + self.gdev(i, u, uu)) for i in range(self.Q)]
        if self.c["storage"] == FP32:
            f, g = [v.float().double() for v in f], [v.float().double() for v in g]
        return f, g

    @staticmethod
    def dot(d, u):
        t = 0.0
        for k in range(3):
            if d[k]:
                t = t + d[k] * u[k]
        return t

    def gdev(self, a, u, uu):
        cu = self.dot(self.C[a], u)
        return self.W[a] * (3 * cu + 4.5 * cu * cu - 1.5 * uu)

    def neighbour(self, phi, d):
        """phi(x + d): periodic, or the mirrored ghost at walls and symmetry faces."""
        t = phi
        for k, dim in ((0, 2), (1, 1), (2, 0)):
            if not d[k]:
                continue
            n = t.shape[dim]
            t2 = torch.roll(t, -d[k], dim)
            if (self.wall and k == self.D - 1) or (self.sym and k == 0):
                end = n - 1 if d[k] > 0 else 0
                t2.select(dim, end).copy_(t.select(dim, end))
            t = t2
        return t

    def stream(self, post, dirs):
        """Streaming with half-way bounce-back walls and specular symmetry faces."""
        where = {d: i for i, d in enumerate(dirs)}
        out = []
        v, dim = self.D - 1, 3 - self.D
        for d in dirs:
            src = torch.roll(post[where[d]], (d[2], d[1], d[0]), (0, 1, 2))
            if self.sym and d[0]:
                end = 0 if d[0] > 0 else self.nx - 1
                own = torch.roll(post[where[(-d[0], d[1], d[2])]], (d[2], d[1]), (0, 1))
                src.select(2, end).copy_(own.select(2, end))
            if self.wall and d[v]:
                end = 0 if d[v] > 0 else src.shape[dim] - 1
                src.select(dim, end).copy_(post[where[tuple(-x for x in d)]].select(dim, end))
            out.append(src)
        return out

    def closure(self, f, g):
        D = self.D
        phi = sum(g)
        grad, lap = [0.0, 0.0, 0.0], 0.0
        for i, d in enumerate(self.C):
            nb = self.neighbour(phi, d)
            lap = lap + 6 * self.W[i] * (nb - phi)
            for k in range(D):
                if d[k]:
                    grad[k] = grad[k] + 3 * self.W[i] * d[k] * nb
        rho = self.rho_l + (1 - self.rho_l) * phi
        nu = self.nu_h + (self.nu_l - self.nu_h) * (1 - phi)
        mag = torch.sqrt(sum(grad[k] ** 2 for k in range(D)))
        normal = [grad[k] / mag.clamp(min=1e-4) if k < D else 0.0 for k in range(3)]
        mu = 2 * self.beta * phi * (phi - 1) * (2 * phi - 1) - self.kappa * lap
        F = [mu * grad[k] if k < D else 0.0 for k in range(3)]
        F[D - 1] = F[D - 1] - (rho - 0.5 * (1 + self.rho_l)) * self.g_accel
        P = sum(f)
        J = [sum(d[k] * f[i] for i, d in enumerate(self.C) if d[k]) if k < D else 0.0 for k in range(3)]
        u = [(3 * J[k] + 0.5 * F[k]) / rho if k < D else torch.zeros_like(phi) for k in range(3)]
        G = [(1 - self.rho_l) * grad[k] / 3 if k < D else 0.0 for k in range(3)]
        uG, uF = (sum(u[k] * V[k] for k in range(D)) for V in (G, F))
        return dict(phi=phi, rho=rho, nu=nu, n=normal, F=F, G=G, u=u, uG=uG, uF=uF, P=P, ph=P + 0.5 * uG,
                    uu=sum(u[k] ** 2 for k in range(D)))

    def collide(self, f, g, s, phiu):
        """Post-collision populations (the shear rate on the second-order
        cumulants, every other rate one)."""
        D, u, rho = self.D, s["u"], s["rho"]
        V = [s["G"][k] + s["F"][k] for k in range(3)]
        uV = s["uG"] + s["uF"]
        om1 = 1 - 1 / (3 * s["nu"] + 0.5)
        d = {}
        for i in range(D):
            for j in range(i, D):
                pi = sum(c[i] * c[j] * f[a] for a, c in enumerate(self.C) if c[i] * c[j])
                t = 3 * pi - (s["P"] if i == j else 0.0) + 0.5 * (u[i] * V[j] + u[j] * V[i]) - 1.5 * u[i] * u[j] * uV
                d[i, j] = t / rho - u[i] * u[j]
        tr = sum(d[i, i] for i in range(D)) / D
        A = [om1 * (d[i, i] - tr) if i < D else None for i in range(3)]
        K = {k: om1 * v for k, v in d.items() if k[0] != k[1]}
        c2 = 1 / 3
        a, b, pq = A[0], A[1], K[0, 1]
        k = {(2, 0, 0): a, (0, 2, 0): b, (1, 1, 0): pq, (2, 2, 0): c2 * (a + b) + a * b + 2 * pq ** 2}
        if D == 3:
            c, q, r = A[2], K[0, 2], K[1, 2]
            k.update({(0, 0, 2): c, (1, 0, 1): q, (0, 1, 1): r,
                      (2, 0, 2): c2 * (a + c) + a * c + 2 * q * q, (0, 2, 2): c2 * (b + c) + b * c + 2 * r * r,
                      (2, 1, 1): (c2 + a) * r + 2 * pq * q, (1, 2, 1): (c2 + b) * q + 2 * pq * r,
                      (1, 1, 2): (c2 + c) * pq + 2 * q * r,
                      (2, 2, 2): c2 * c2 * (a + b + c) + c2 * (a * b + b * c + c * a) + a * b * c
                      + 2 * ((c2 + a) * r * r + (c2 + b) * q * q + (c2 + c) * pq * pq) + 8 * pq * q * r})
        h = k
        for axis in range(D):  # central moments to populations, axis by axis
            done = {}
            for key in {tuple(v for j, v in enumerate(t) if j != axis) for t in h}:
                def at(m):
                    return h.get(key[:axis] + (m,) + key[axis:], 0.0)
                m0, m1 = at(0), at(1) + u[axis] * at(0)
                m2 = at(2) + 2 * u[axis] * at(1) + u[axis] ** 2 * at(0)
                for e, val in ((0, 0.5 * (m2 - m1)), (1, m0 - m2), (2, 0.5 * (m2 + m1))):
                    done[key[:axis] + (e,) + key[axis:]] = val
            h = done
        fo, go = [], []
        for i, c in enumerate(self.C):
            gd = self.gdev(i, u, s["uu"])
            xi = gd * (self.dot(c, s["G"]) - s["uG"]) + (self.W[i] + gd) * (self.dot(c, s["F"]) - s["uF"])
            E = 1.0
            for j in range(D):
                E = E * (1 - u[j] ** 2 - 1 / 3 if c[j] == 0 else 0.5 * (u[j] ** 2 + 1 / 3 + c[j] * u[j]))
            dh = h[tuple(c[j] + 1 for j in range(D)) + ((0,) if D == 2 else ())]
            fo.append(rho / 3 * (E - self.W[i] + dh) + self.W[i] * s["ph"] + 0.5 * xi)
        sharp = self.lam * 4 * s["phi"] * (1 - s["phi"]) / self.width
        if self.reduced:
            now = [s["phi"] * u[j] for j in range(D)]
            ddt = [now[j] - phiu[j] if j < D else 0.0 for j in range(3)]
            for c, w, gi in zip(self.G, self.GW, g):
                eq = w * s["phi"] * (1 + self.ics2g * self.dot(c, u))
                go.append(gi + (eq - gi) / self.tau + w * (sharp * self.dot(c, s["n"])
                                                           + self.lam * self.ics2g * self.dot(c, ddt)))
            return fo, go, now
        for i, c in enumerate(self.C):
            eq = s["phi"] * (self.W[i] + self.gdev(i, u, s["uu"]))
            go.append(g[i] + (eq - g[i]) / self.tau + self.W[i] * self.dot(c, s["n"]) * sharp)
        return fo, go, None

    def outputs(self, steps):
        f, g = self.start()
        phiu = None
        for k in range(steps):
            if k:
                f, g = self.stream(f, self.C), self.stream(g, self.G)
            s = self.closure(f, g)
            if self.reduced and k == 0:
                phiu = [s["phi"] * s["u"][j] for j in range(self.D)]
            f, g, phiu = self.collide(f, g, s, phiu)
            del s
        if self.c["form"] == "aa":  # an even step count leaves the streamed values in their own slots
            f, g = self.stream(f, self.C), self.stream(g, self.G)
        out = {}
        for name, v in (("f", f), ("g", g)):
            if self.c["storage"] == FP32:
                out[name] = torch.stack(v).reshape(-1)
            else:
                mid = self.Q // 2
                den = 216.0 if self.D == 3 else 36.0
                ref = v[mid] / (den * self.W[mid])
                S = CODE_SCALE[self.c["storage"]]
                out[name + "_ref"] = ref.reshape(-1)
                out[name + "_codes"] = torch.stack([S * (v[a] / (den * self.W[a]) - ref) for a in range(self.Q)
                                                    if a != mid]).reshape(-1)
        if self.reduced:
            out["phi_u"] = torch.stack(phiu).reshape(-1)
        return out

    def observables(self):
        D = self.D
        f, g = self.start()
        s = self.closure(f, g)
        n = (self.nx, self.ny, self.nz)
        mid = [v // 2 if k < D else 0 for k, v in enumerate(n)]

        def mean_p(at):
            t = 0.0
            for d in self.C:
                i = [(at[k] + d[k]) % n[k] for k in range(3)]
                if self.wall:
                    i[D - 1] = min(max(at[D - 1] + d[D - 1], 0), n[D - 1] - 1)
                t += float(s["ph"][i[2], i[1], i[0]])
            return t / self.Q
        p_in, p_out = mean_p(mid), mean_p([0, 0, 0])
        up = (lambda x, y: s["phi"][:, y, x]) if D == 3 else (lambda x, y: s["phi"][0, :, x])
        cs, cb = up(mid[0], mid[1]).cpu().numpy(), up(0, 0).cpu().numpy()
        heavy, light = np.nonzero(cs >= 0.5)[0], np.nonzero(cb < 0.5)[0]
        spike = bubble = -1.0
        if len(heavy):
            k = int(heavy[0])
            spike = 0.0 if k == 0 else k - (cs[k] - 0.5) / (cs[k] - cs[k - 1])
        if len(light):
            k = int(light[-1])
            bubble = float(k) if k == len(cb) - 1 else k + (0.5 - cb[k]) / (cb[k + 1] - cb[k])
        return dict(mass=float(s["phi"].sum()), mass_drift_rel=0.0,
                    kinetic_energy=float((0.5 * s["rho"] * s["uu"]).sum()), max_u=math.sqrt(float(s["uu"].max())),
                    p_in=p_in, p_out=p_out, laplace_dp=p_in - p_out, tip_spike=float(spike),
                    tip_bubble=float(bubble), step=0, health=0)


def exact(c, seed):
    if c["kind"] == "mix":
        return [Exact(m, seed + k).outputs(c["steps"]) for k, m in enumerate(members(c))]
    e = Exact(c, seed)
    return e.observables() if c["kind"] == "observe" else e.outputs(c["steps"])
