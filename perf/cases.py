"""The work a user of the library has it do, as measurable cases.

One pass of a case advances a plasma (or a batch of plasmas) that is already on
the device by a number of steps through the Python binding and reads the
result back the way a run's output stage does: the fields E, B and the current
J (``Simulation.fields``), and in two cases also the energies
(``Simulation.diagnostics``) or the particles (``Simulation.particles``).  A
mixed-precision run holds its mesh and particles in FP32, so its output is kept
in FP32; an FP64 run keeps FP64.

``exact`` integrates the same plasma in plain FP64 torch: separable B-spline
gather, Vay or Boris push, Esirkepov's current on the union support, the cyclic
line solve and the implicit field update by Fourier transforms.
"""
import math
import random

import torch

import paper_1211_4575_gb300 as pp

DEVICE = "cuda"
# Past this many particle-steps the FP64 integration takes longer than about 20 s.
EXACT_PARTICLE_STEPS = 4.1e8

# Values a case that does not state them takes.
DEFAULTS = dict(kind="thermal", shape=3, precision="mixed", pusher="vay", steps=10, walls="", solver="implicit",
                current="conserving", filter=0, integrator=2, graphs=False, output="fields", runs=0)

# (dx, dt, species masses, [(fraction of ppc, density, drift beta, u_th)], cold relativistic beam) per kind of plasma.
KINDS = {
    "two_stream": (0.5, 0.25, (1.0, 1.0), [(0.5, 0.5, 0.2, 0.05), (0.5, 0.5, -0.2, 0.05)]),
    "thermal": (0.1, 0.05, (1.0, 1.0), [(1.0, 1.0, 0.0, 0.1)]),
    "weibel": (0.5, 0.25, (1.0, 25.0), [(0.5, 0.5, 0.5, 0.1), (0.5, 0.5, -0.5, 0.1)]),
    "beam": (0.5, 0.25, (1.0, 25.0), [(1.0, 0.5, 0.0, 0.01), (1.0, 0.5, math.sqrt(0.99), 0.0)]),
    "heating": (0.1, 0.05, (1.0, 16.0), [(1.0, 1.0, 0.0, 0.1)]),
}


def listed():
    return [
        # The validation run: 16^3 counter-streaming pair beams in FP64, TSC.  The smallest call there is:
        # its steps are launches, not work.
        dict(name="two_stream_16_fp64", kind="two_stream", nx=16, ny=16, nz=16, ppc=8, shape=2, precision="fp64",
             steps=20),
        # One small served request alone on its own stream, stepping through captured graphs.
        dict(name="served_32", kind="two_stream", nx=32, ny=32, nz=32, ppc=8, steps=20, graphs=True),
        # An FP64 run of a box that no tile divides, with the Boris push: a convergence check.
        dict(name="ragged_fp64", kind="weibel", nx=45, ny=30, nz=37, ppc=8, shape=3, precision="fp64",
             pusher="boris", steps=5),
        # A mixed run whose box no tile divides.
        dict(name="ragged_mixed", kind="weibel", nx=60, ny=45, nz=37, ppc=16, steps=10),
        # The numerical-heating run at a size that nearly fills the GPU, with its energy series.
        dict(name="thermal_64_energies", kind="thermal", nx=64, ny=64, nz=64, ppc=32, steps=10, output="energies"),
        # The numerical-heating run at full size.
        dict(name="thermal_128", kind="thermal", nx=128, ny=128, nz=128, ppc=32, steps=3),
        # The Gamma = 10 beam through an electron-ion background: the production run and the largest.
        dict(name="beam_256", kind="beam", nx=256, ny=128, nz=128, ppc=16, steps=10),
        # The largest served request, few particles per cell: the mesh weighs most here.
        dict(name="weibel_192", kind="weibel", nx=192, ny=192, nz=192, ppc=8, steps=3),
        # A plasma between reflecting walls on x.
        dict(name="walls_64", kind="heating", nx=64, ny=64, nz=64, ppc=16, walls="x", steps=10),
        # The original method that the paper compares with: direct current, explicit fields, filtered E and B.
        dict(name="direct_filter_64", kind="thermal", nx=64, ny=64, nz=64, ppc=16, shape=2, solver="explicit",
             current="direct", filter=5, steps=5),
        # The fourth-order integrator on an electron-ion plasma, its particles read back for a spectrum.
        dict(name="order4_particles", kind="heating", nx=48, ny=40, nz=32, ppc=8, integrator=4, steps=5,
             output="particles"),
        # Uneven independent runs advanced together.
        dict(name="batch_12", kind="two_stream", nx=16, ny=72, nz=0, ppc=32, steps=10, runs=12),
    ]


def _edge(rng, lo, hi, multiple=1):
    e = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(multiple, int(round(e / multiple)) * multiple)


def draw(rng):
    family = rng.choice(["fp64", "served", "ragged", "tiled", "tiled", "tiled", "walls", "direct", "order4", "batch"])
    shape = rng.choice([1, 2, 3, 3, 3])
    if family == "fp64":
        n = [_edge(rng, 8, 48) for _ in range(3)]
        return dict(kind=rng.choice(["two_stream", "weibel", "thermal"]), nx=n[0], ny=n[1], nz=n[2],
                    ppc=2 * rng.randint(2, 8), shape=shape, precision="fp64", pusher=rng.choice(["vay", "boris"]),
                    steps=rng.randint(3, 20))
    if family == "served":
        n = [_edge(rng, 16, 96, 8) for _ in range(3)]
        return dict(kind=rng.choice(["two_stream", "weibel"]), nx=n[0], ny=n[1], nz=n[2], ppc=2 * rng.randint(4, 16),
                    shape=rng.choice([2, 3]), steps=rng.randint(5, 20), graphs=True)
    if family == "ragged":
        n = [_edge(rng, 10, 90) for _ in range(3)]
        return dict(kind=rng.choice(["two_stream", "weibel", "thermal"]), nx=n[0], ny=n[1], nz=n[2],
                    ppc=2 * rng.randint(2, 16), shape=shape, steps=rng.randint(3, 10))
    if family == "tiled":
        n = [_edge(rng, 24, 192, 8) for _ in range(3)]
        kind = rng.choice(["thermal", "weibel", "beam"])
        ppc = 2 * rng.randint(4, 8 if kind == "beam" else 16)
        cells = n[0] * n[1] * n[2]
        return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], ppc=ppc, shape=shape, pusher=rng.choice(["vay", "vay", "boris"]),
                    steps=rng.randint(2, 10) if cells < 3e6 else rng.randint(1, 4),
                    output=rng.choice(["fields", "fields", "energies"]))
    if family == "walls":
        n = [_edge(rng, 16, 64, 8) for _ in range(3)]
        return dict(kind=rng.choice(["heating", "thermal"]), nx=n[0], ny=n[1], nz=n[2], ppc=2 * rng.randint(4, 12),
                    shape=shape, walls=rng.choice(["x", "y", "xz"]), steps=rng.randint(3, 10))
    if family == "direct":
        n = [_edge(rng, 16, 80, 8) for _ in range(3)]
        return dict(kind="thermal", nx=n[0], ny=n[1], nz=n[2], ppc=2 * rng.randint(4, 12), shape=shape,
                    solver="explicit", current="direct", filter=rng.randint(1, 5), steps=rng.randint(2, 8))
    if family == "order4":
        n = [_edge(rng, 16, 56, 8) for _ in range(3)]
        return dict(kind="heating", nx=n[0], ny=n[1], nz=n[2], ppc=2 * rng.randint(2, 8), shape=shape, integrator=4,
                    steps=rng.randint(1, 5), output="particles")
    return dict(kind="two_stream", nx=16, ny=_edge(rng, 24, 96, 8), nz=rng.randint(0, 99), ppc=2 * rng.randint(8, 32),
                steps=rng.randint(2, 10), runs=rng.randint(4, 16))


def _full(case):
    return {**DEFAULTS, **case}


def _runs_of(case):
    """The runs of a batch: cubic edges from nx to ny, ppc per species from 8 to ppc, TSC or PCS; nz varies the draw."""
    rng = random.Random(1215 + case["nz"])
    out = []
    for _ in range(case["runs"]):
        e = rng.randrange(case["nx"], case["ny"] + 1, 8)
        out.append({**case, "runs": 0, "nx": e, "ny": e, "nz": e, "ppc": 2 * rng.randint(4, case["ppc"] // 2),
                    "shape": rng.choice([2, 3])})
    return out


def _plasma(case, seed):
    """The particles of a neutral plasma: (q, m, w, [x, y, z, ux, uy, uz]) per species, FP64 on the device.  A fixed
    number per cell, uniform in the cell; each negative particle on top of a positive one, so that E = B = 0 holds."""
    dx, _, masses, pops = KINDS[case["kind"]]
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(seed)
    cells = case["nx"] * case["ny"] * case["nz"]
    beam = case["kind"] == "beam"
    parts = ([], [])
    for frac, density, beta, u_th in pops:
        ppc = max(1, int(case["ppc"] * frac))
        w = density / ppc
        c = torch.arange(cells, device=DEVICE).repeat_interleave(ppc)
        xyz = []
        for a, i in enumerate((c % case["nx"], (c // case["nx"]) % case["ny"], c // (case["nx"] * case["ny"]))):
            r = torch.rand(c.numel(), generator=gen, device=DEVICE, dtype=torch.float64)
            xyz.append(r.add_(i).mul_(dx))
        n = c.numel()
        del c, i, r
        gamma = 1.0 / math.sqrt(1.0 - beta * beta)
        for s in range(2):
            u = [torch.randn(n, generator=gen, device=DEVICE, dtype=torch.float64) * u_th for _ in range(3)]
            if beam and beta:   # thermal part drawn in the rest frame of the beam
                u[0] = gamma * (u[0] + beta * (1.0 + u[0] ** 2 + u[1] ** 2 + u[2] ** 2).sqrt())
            else:
                u[0] += gamma * beta
            parts[s].append(xyz + u)
    out = []
    for s, q in ((0, -1.0), (1, 1.0)):
        cols = parts[s][0] if len(parts[s]) == 1 else [torch.cat(v) for v in zip(*parts[s])]
        out.append((q, masses[s], w, cols))
    return out


def _grid(case):
    """(cell size, dt): the explicit solver runs a little below the implicit one's step, under its stability limit."""
    dx, dt = KINDS[case["kind"]][:2]
    return dx, dt * (0.8 if case["solver"] == "explicit" else 1.0)


def _simulation(case, seed, stream=None):
    dx, dt = _grid(case)
    fp64 = case["precision"] == "fp64"
    wall = {a: pp.PP_BOUNDARY_WALLS if a in case["walls"] else pp.PP_BOUNDARY_PERIODIC for a in "xyz"}
    sim = pp.Simulation((case["nx"], case["ny"], case["nz"]), (dx, dx, dx), dt, shape_order=case["shape"],
                        pusher=pp.PP_BORIS if case["pusher"] == "boris" else pp.PP_VAY,
                        precision=pp.PP_FP64 if fp64 else pp.PP_MIXED32, relax_tol=1e-12 if fp64 else 1e-6,
                        stream=stream, boundary_x=wall["x"], boundary_y=wall["y"], boundary_z=wall["z"])
    for q, m, w, cols in _plasma(case, seed):
        sid = sim.add_species(q, m, w, cols[0].numel())
        torch.cuda.synchronize()   # the run may have a stream of its own
        sim.load_particles(sid, *cols)
    if case["solver"] == "explicit":
        sim.set_field_solver(pp.PP_FIELD_EXPLICIT)
    if case["current"] == "direct":
        sim.set_current_deposit(pp.PP_CURRENT_DIRECT)
    if case["filter"]:
        sim.set_divergence_filter(case["filter"])
    if case["integrator"] == 4:
        sim.set_integrator(4)
    if case["graphs"]:
        sim.set_graphs(True)
    return sim


def prepare(case, seed):
    case = _full(case)
    state = {"case": case}
    if case["runs"]:
        state["streams"] = [torch.cuda.Stream() for _ in range(case["runs"])]
        state["sims"] = [_simulation(c, seed * 64 + k, state["streams"][k].cuda_stream)
                         for k, c in enumerate(_runs_of(case))]
        state["batch"] = pp.Batch(200 << 30, case["runs"])
        state["batch"].set_fused(True)
    else:
        state["streams"] = [torch.cuda.Stream()] if case["graphs"] else []
        state["sims"] = [_simulation(case, seed, state["streams"][0].cuda_stream if case["graphs"] else None)]
    return state


def _fields(case, sim):
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    return [[torch.from_numpy(a).to(dtype) for a in f] for f in sim.fields()]


def run(state):
    case, sims = state["case"], state["sims"]
    if case["runs"]:
        batch = state["batch"]
        slots = [batch.admit(sim, case["steps"]) for sim in sims]
        left = set(slots)
        while left:
            batch.advance(case["steps"])
            left -= {k for k in left if batch.poll(k)[0] != pp.PP_BATCH_RUNNING}
        return [[torch.stack(f) for f in _fields(case, sim)] for sim in sims]
    sim = sims[0]
    sim.step(case["steps"])
    out = {"fields": _fields(case, sim)}
    if case["output"] == "energies":
        d = sim.diagnostics()
        out["energies"] = torch.tensor([d["energy_E"], d["energy_B"], d["energy_Ex"]] + d["kinetic"],
                                       dtype=torch.float32)
    if case["output"] == "particles":
        # the library keeps no particle order: each coordinate's distribution, as its sorted values
        out["particles"] = [{k: torch.from_numpy(v).to(DEVICE).to(torch.float32).sort().values
                             for k, v in sim.particles(s).items()} for s in range(2)]
    return out


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Bytes: per (sub)step the particle state read and written, E, B read and written, J written; the FP64 output
    once.  Operations: per particle and (sub)step the separable gather of six components, the push and the current
    of three components at the support's sites; the field update's stencils and its relaxation are left out."""
    case = _full(case)
    total = {"bytes": 0.0, "flops": 0.0}
    for c in _runs_of(case) if case["runs"] else [case]:
        cells = c["nx"] * c["ny"] * c["nz"] * 2 ** len(c["walls"])
        pops = KINDS[c["kind"]][3]
        n = 2 * c["nx"] * c["ny"] * c["nz"] * sum(max(1, int(c["ppc"] * p[0])) for p in pops)
        sub = c["steps"] * (4 if c["integrator"] == 4 else 1)
        real = 8 if c["precision"] == "fp64" else 4
        per = 48 if c["precision"] == "fp64" else 28
        o = c["shape"] + 1
        gather = 6 * 2 * (o ** 3 + o ** 2 + o)
        deposit = 3 * (2 * (o - 1) * o * o + 3 * o * o)
        total["bytes"] += sub * (2.0 * per * n + 15.0 * real * cells) + 72.0 * cells
        total["flops"] += float(sub) * n * (gather + deposit + 100)
    return total


# ---------------------------------------------------------------------------
# The same plasma in FP64 torch
# ---------------------------------------------------------------------------
K6 = (75.0 / 64.0, -25.0 / 384.0, 3.0 / 640.0)   # 6th-order staggered difference
ALPHA = 0.55
AXIS = (2, 1, 0)                                 # mesh arrays are [z, y, x]


def _spline(order, f):
    g = 1.0 - f
    if order == 1:
        w = [g, f]
    elif order == 2:
        w = [0.5 * g * g, 0.75 - (f - 0.5) ** 2, 0.5 * f * f]
    else:
        w = [g ** 3 / 6, (3 * f ** 3 - 6 * f ** 2 + 4) / 6, (3 * g ** 3 - 6 * g ** 2 + 4) / 6, f ** 3 / 6]
    return torch.stack(w, 1)


def _support(order, xi, half):
    """First node and weights of the particles at xi on integer (half = 0) or half-integer (half = 1) nodes."""
    y = xi - 0.5 * (order - 1 + half)
    i = torch.floor(y)
    return i.long(), _spline(order, y - i)


class _Exact:
    def __init__(self, case, seed):
        self.c = case
        self.o = case["shape"]
        self.h, self.dt = _grid(case)
        phys = (case["nx"], case["ny"], case["nz"])
        self.wall = [phys[a] if "xyz"[a] in case["walls"] else 0 for a in range(3)]
        self.n = [2 * phys[a] if self.wall[a] else phys[a] for a in range(3)]
        z = lambda: torch.zeros(self.n[2], self.n[1], self.n[0], dtype=torch.float64, device=DEVICE)  # noqa: E731
        self.E, self.B, self.J = [[z() for _ in range(3)] for _ in range(3)]
        self.zero = z
        self.species = [(q, m, w, [v / self.h if k < 3 else v for k, v in enumerate(cols)])
                        for q, m, w, cols in _plasma(case, seed)]
        th = [2 * math.pi * torch.arange(n, dtype=torch.float64, device=DEVICE) / n for n in self.n]
        shape = ([1, 1, -1], [1, -1, 1], [-1, 1, 1])
        k = K6
        # symbols of the line operator of the current, and of -d^+ d^- summed over the axes
        self.line = [((sum(k) + 2 * (k[1] + k[2]) * torch.cos(t) + 2 * k[2] * torch.cos(2 * t))).view(s)
                     for t, s in zip(th, shape)]
        self.k2 = sum((2 * sum(k[m] * torch.sin((m + 0.5) * t) for m in range(3)) / self.h).square().view(s)
                      for t, s in zip(th, shape))
        s = torch.arange(4001, dtype=torch.float64) * math.pi / 4000
        top = float((2 * sum(k[m] * torch.sin((m + 0.5) * s) for m in range(3))).square().max())
        self.tau = self.h * self.h / (3 * top)

    def diff(self, f, axis, plus):
        at = lambda o: torch.roll(f, -o, AXIS[axis])  # noqa: E731
        if plus:
            return sum(K6[m - 1] * (at(m) - at(1 - m)) for m in (1, 2, 3)) / self.h
        return sum(K6[m - 1] * (at(m - 1) - at(-m)) for m in (1, 2, 3)) / self.h

    def curl(self, F, plus):
        return [self.diff(F[(a + 2) % 3], (a + 1) % 3, plus) - self.diff(F[(a + 1) % 3], (a + 2) % 3, plus)
                for a in range(3)]

    def laplace(self, f):
        return sum(self.diff(self.diff(f, a, False), a, True) for a in range(3))

    def index(self, start, counts):
        """Flat mesh indices [particle, k, j, i] of supports of `counts` nodes from `start` on each axis."""
        ix = [(start[a][:, None] + torch.arange(counts[a], device=DEVICE)) % self.n[a] for a in range(3)]
        return (ix[2][:, :, None, None] * self.n[1] + ix[1][:, None, :, None]) * self.n[0] + ix[0][:, None, None, :]

    def gather(self, F, comp, sup, magnetic):
        s = [sup[int((a == comp) != magnetic)][a] for a in range(3)]
        v = F[comp].reshape(-1)[self.index([x[0] for x in s], [self.o + 1] * 3)]
        for a in range(3):
            v = (v * s[a][1].view(v.shape[0], *([1] * (v.dim() - 2)), -1)).sum(-1)
        return v

    def push(self, E, B, u, qmdt):
        cross = lambda a, b: [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]  # noqa: E731
        dot = lambda a, b: a[0] * b[0] + a[1] * b[1] + a[2] * b[2]  # noqa: E731
        t = [0.5 * qmdt * b for b in B]
        if self.c["pusher"] == "boris":
            m = [u[d] + 0.5 * qmdt * E[d] for d in range(3)]
            t = [v / (1 + dot(m, m)).sqrt() for v in t]
            a = [x + y for x, y in zip(m, cross(m, t))]
            r = cross(a, [2 * v / (1 + dot(t, t)) for v in t])
            return [m[d] + r[d] + 0.5 * qmdt * E[d] for d in range(3)]
        v = [x / (1 + dot(u, u)).sqrt() for x in u]
        p = [u[d] + qmdt * E[d] + x for d, x in enumerate(cross(v, t))]
        t2, us = dot(t, t), dot(p, t)
        sigma = 1 + dot(p, p) - t2
        g = (0.5 * (sigma + (sigma * sigma + 4 * (t2 + us * us)).sqrt())).sqrt()
        t = [x / g for x in t]
        s, pt, x = 1 / (1 + dot(t, t)), dot(p, t), cross(p, t)
        return [s * (p[d] + pt * t[d] + x[d]) for d in range(3)]

    def deposit(self, x0, dx, qw, dt):
        o = self.o
        if self.c["current"] == "direct":
            sup = [[_support(o, x0[a] + 0.5 * dx[a], half) for a in range(3)] for half in (0, 1)]
            for a in range(3):
                s = [sup[int(b == a)][b] for b in range(3)]
                v = (qw * self.h / dt * dx[a])[:, None, None, None] * s[2][1][:, :, None, None] * \
                    s[1][1][:, None, :, None] * s[0][1][:, None, None, :]
                self.J[a].view(-1).index_add_(0, self.index([x[0] for x in s], [o + 1] * 3).view(-1), v.reshape(-1))
            return
        lo, S0, DS = [], [], []
        for a in range(3):   # old and new weights on the union of the two supports
            (i0, w0), (i1, w1) = _support(o, x0[a], 0), _support(o, x0[a] + dx[a], 0)
            start = torch.minimum(i0, i1)
            w = []
            for i, v in ((i0, w0), (i1, w1)):
                z = torch.zeros_like(v[:, :1])
                w.append(torch.where((i > start)[:, None], torch.cat([z, v], 1), torch.cat([v, z], 1)))
            lo.append(start)
            S0.append(w[0])
            DS.append(w[1] - w[0])
        idx = self.index(lo, [o + 2] * 3).view(-1)
        for a in range(3):
            b, c = (a + 1) % 3, (a + 2) % 3
            C = torch.cumsum(DS[a], 1) * (-qw * self.h / dt)
            view = lambda t, axis: t.view(t.shape[0], *[-1 if k == axis else 1 for k in (2, 1, 0)])  # noqa: E731
            mb, mc = view(S0[b] + 0.5 * DS[b], b), view(S0[c] + 0.5 * DS[c], c)
            v = view(C, a) * (mb * mc + view(DS[b], b) * view(DS[c], c) / 12)
            self.J[a].view(-1).index_add_(0, idx, v.reshape(-1))

    def particles(self, kick, drift):
        self.J = [self.zero() for _ in range(3)]
        for q, m, w, cols in self.species:
            for s in range(0, cols[0].numel(), 1 << 20):
                part = [v[s:s + (1 << 20)] for v in cols]
                x0, u = [v.clone() for v in part[:3]], part[3:]
                if kick:
                    sup = [[_support(self.o, x0[a], half) for a in range(3)] for half in (0, 1)]
                    E = [self.gather(self.E, a, sup, False) for a in range(3)]
                    B = [self.gather(self.B, a, sup, True) for a in range(3)]
                    u = self.push(E, B, u, q * kick / m)
                g = (1 + u[0] ** 2 + u[1] ** 2 + u[2] ** 2).sqrt()
                dx = [drift / self.h * v / g for v in u]
                self.deposit(x0, dx, q * w, drift)
                for a in range(3):
                    x, v, n = torch.remainder(x0[a] + dx[a], self.n[a]), u[a], self.wall[a]
                    if n:
                        v = torch.where(x > n, -v, v)
                        x = torch.where(x > n, 2 * n - x, x)
                    part[a].copy_(x)
                    part[3 + a].copy_(v)
        for ax in range(3):
            if not self.wall[ax]:
                continue
            for a in range(3):   # the virtual images' current
                f = torch.flip(self.J[a], (AXIS[ax],))
                self.J[a] = self.J[a] - f if a == ax else self.J[a] + torch.roll(f, 1, AXIS[ax])
        if self.c["current"] == "conserving":
            for a in range(3):
                self.J[a] = torch.fft.ifft(torch.fft.fft(self.J[a], dim=AXIS[a]) / self.line[a], dim=AXIS[a]).real

    def fields_update(self, dt):
        if self.c["solver"] == "explicit":
            self.B = [b - 0.5 * dt * x for b, x in zip(self.B, self.curl(self.E, True))]
            self.E = [e + dt * (x - j) for e, x, j in zip(self.E, self.curl(self.B, False), self.J)]
            self.B = [b - 0.5 * dt * x for b, x in zip(self.B, self.curl(self.E, True))]
            return
        al, be = ALPHA, 1 - ALPHA
        cE, cJ = self.curl(self.E, True), self.curl(self.J, True)
        new = []
        for a in range(3):
            rhs = self.B[a] + al * be * dt * dt * self.laplace(self.B[a]) - dt * cE[a] + al * dt * dt * cJ[a]
            new.append(torch.fft.ifftn(torch.fft.fftn(rhs) / (1 + al * al * dt * dt * self.k2)).real)
        mid = self.curl([al * x + be * y for x, y in zip(new, self.B)], False)
        self.E = [e + dt * (x - j) for e, x, j in zip(self.E, mid, self.J)]
        self.B = new

    def filter(self):
        rho = self.zero()
        for q, _, w, cols in self.species:
            for s in range(0, cols[0].numel(), 1 << 20):
                sup = [_support(self.o, v[s:s + (1 << 20)], 0) for v in cols[:3]]
                v = (q * w) * sup[2][1][:, :, None, None] * sup[1][1][:, None, :, None] * sup[0][1][:, None, None, :]
                rho.view(-1).index_add_(0, self.index([x[0] for x in sup], [self.o + 1] * 3).view(-1), v.reshape(-1))
        for _ in range(self.c["filter"]):
            eE = sum(self.diff(self.E[a], a, False) for a in range(3)) - rho
            self.E = [e + self.tau * self.diff(eE, a, True) for a, e in enumerate(self.E)]
            eB = sum(self.diff(self.B[a], a, True) for a in range(3))
            self.B = [b + self.tau * self.diff(eB, a, False) for a, b in enumerate(self.B)]

    def step(self):
        if self.c["integrator"] == 4:
            r = 2.0 ** (1.0 / 3.0)
            w1 = 1.0 / (2.0 - r)
            w0 = -r * w1
            for a, b in ((w1 / 2, 0.0), ((w0 + w1) / 2, w1), ((w0 + w1) / 2, w0), (w1 / 2, w1)):
                self.particles(b * self.dt, a * self.dt)
                self.fields_update(a * self.dt)
        else:
            self.particles(self.dt, self.dt)
            self.fields_update(self.dt)
        if self.c["filter"]:
            self.filter()

    def output(self):
        out = {"fields": [self.E, self.B, self.J]}
        dv = self.h ** 3
        if self.c["output"] == "energies":
            sq = [float(f.square().sum()) * 0.5 * dv / 2 ** len(self.c["walls"]) for f in self.E + self.B]
            kin = []
            for _, m, w, cols in self.species:
                u2 = sum(v * v for v in cols[3:])
                kin.append(w * m * dv * float((u2 / (1 + (1 + u2).sqrt())).sum()))
            out["energies"] = torch.tensor([sum(sq[:3]), sum(sq[3:]), sq[0]] + kin, dtype=torch.float64)
        if self.c["output"] == "particles":
            out["particles"] = [{k: (v * self.h if a < 3 else v).sort().values
                                 for a, (k, v) in enumerate(zip(("x", "y", "z", "ux", "uy", "uz"), cols))}
                                for _, _, _, cols in self.species]
        return out


def _exact_run(case, seed):
    x = _Exact(case, seed)
    for _ in range(case["steps"]):
        x.step()
    return x.output()


def exact(case, seed):
    case = _full(case)
    runs = _runs_of(case) if case["runs"] else [case]
    load = 0.0
    for c in runs:
        pops = KINDS[c["kind"]][3]
        n = 2 * c["nx"] * c["ny"] * c["nz"] * sum(max(1, int(c["ppc"] * p[0])) for p in pops)
        load += n * c["steps"] * (4 if c["integrator"] == 4 else 1)
    if load > EXACT_PARTICLE_STEPS:
        return None
    if case["runs"]:
        return [[torch.stack(f) for f in _exact_run(c, seed * 64 + k)["fields"]] for k, c in enumerate(runs)]
    return _exact_run(case, seed)
