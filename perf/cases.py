"""The work that the framework is timed on: solver runs as its users make them, through the public
classes of ``paper_1710_10569_gb300.clb`` (``Lattice``, ``Batch``, ``Server``, ``Thermal``,
``Lattice3D``, ``Batch3D``), from the smallest lattices of the paper's experiments to the largest of
the benchmark.

A case is a dict of plain values. ``prepare`` builds the handle and its seeded initial state,
``run`` advances it by the case's number of steps (with the convergence checks that a run to steady
state makes) and reads back what a user reads: the macroscopic fields, and the Nusselt number and
residual where the run checks them. A pass starts from where the pass before it ended, as a
simulation does. ``exact`` advances the same initial state in FP64 with plain torch operations:
literal moment sums, shifts and their inverses, independent of the library.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_1710_10569_gb300 import clb
from paper_1710_10569_gb300 import workloads as W

STORAGE = {"f64": W.STORAGE_F64, "f32": W.STORAGE_F32, "f16": W.STORAGE_F16DEV}
BYTES = {"f64": 8, "f32": 4, "f16": 2}

# Node updates that an exact() run stays below (about 20 seconds of FP64 torch operations).
EXACT_LIMIT_2D, EXACT_LIMIT_3D = 4.0e9, 4.0e8


def listed():
    return [
        # The doubly periodic vortex of the accuracy tests: 64 x 64, FP64, stepped 1,000 times and
        # read. The smallest run; every step is a launch's latency.
        dict(name="vortex_64_f64", kind="vortex", nx=64, ny=64, storage="f64", steps=1000, every=0),
        # The paper's Table 1 set-up (60 x 30 cells) with the paper's own walls on the end rows of
        # nodes, run towards steady state with a check every 100 steps.
        dict(name="layer_60x31_wet_f64", kind="layer", nx=60, ny=31, storage="f64", wet=True, Ra=5000.0, steps=2000,
             every=100),
        # The side-heated cavity of the benchmark's steady-state configuration, FP64.
        dict(name="cavity_256_f64", kind="cavity", nx=256, ny=256, storage="f64", Ra=1e5, steps=1000, every=100),
        # A cavity of ordinary size with odd edges and rates of the high-order moments other than 1
        # (the setting of the convergence studies), FP32.
        dict(name="cavity_513x385_f32", kind="cavity", nx=513, ny=385, storage="f32", Ra=1e6, steps=1000, every=100,
             rates=1.2),
        # The benchmark's headline workload: Rayleigh-Benard 2048 x 1024 in FP32, checked every 100
        # steps.
        dict(name="layer_2048x1024_f32", kind="layer", nx=2048, ny=1024, storage="f32", Ra=1e7, steps=1000, every=100),
        # The same in FP64, the reference runs' form.
        dict(name="layer_2048x1024_f64", kind="layer", nx=2048, ny=1024, storage="f64", Ra=1e7, steps=200, every=100),
        # The largest 2-D lattice of the benchmark, half-precision storage (developed flow).
        dict(name="layer_4096x2048_f16", kind="layer", nx=4096, ny=2048, storage="f16", Ra=1e7, steps=1000, every=100),
        # A parameter study: uneven side-heated cavities stepped together, all of them read at the end.
        dict(name="batch_48_f32", kind="batch", count=48, lo=64, hi=512, storage="f32", steps=3000),
        # The request server: small mixed problems submitted together, stepped in chunks of 100 to
        # their step caps, every result fetched.
        dict(name="serve_24_f32", kind="serve", count=24, lo=32, hi=128, storage="f32", steps=1000),
        # A passive scalar in a prescribed velocity field (the D2Q5 equation alone).
        dict(name="scalar_4096_f32", kind="scalar", nx=4096, ny=4096, storage="f32", steps=1500),
        # The benchmark's 3-D Rayleigh-Benard box (D3Q27 + D3Q7).
        dict(name="box_256x256x128_f32", kind="box", nx=256, ny=256, nz=128, storage="f32", Ra=1e7, steps=800),
        # A 3-D parameter study: uneven boxes stepped together.
        dict(name="boxes_12_f32", kind="boxes", count=12, lo=24, hi=128, storage="f32", steps=600),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["vortex", "cavity", "cavity", "layer", "layer", "wet", "batch", "serve", "scalar", "box", "boxes"])
    storage = rng.choice(["f64", "f32", "f32", "f16"])
    budget = 1.2e8 if storage == "f64" else 1.0e9  # node updates of a drawn run
    if kind in ("vortex", "cavity", "layer"):
        nx = _log_int(rng, 32, 4096)
        ny = min(_log_int(rng, 32, 4096), (1 << 23) // nx)
        c = dict(kind=kind, nx=nx, ny=ny, storage=storage)
        if kind != "vortex":
            c["Ra"] = float("%.3g" % math.exp(rng.uniform(math.log(1e4), math.log(1e7))))
        if rng.random() < 0.3:
            c["rates"] = 1.2
        c["every"] = rng.choice([0, 100])
        c["steps"] = max(20, min(1000, int(budget / (nx * ny)) // 10 * 10))
        return c
    if kind == "wet":
        nx, ny = _log_int(rng, 30, 300), _log_int(rng, 16, 160)
        return dict(kind="layer", nx=nx, ny=ny, storage=rng.choice(["f64", "f32"]), wet=True,
                    Ra=float("%.3g" % rng.uniform(2500, 3e4)), steps=1000, every=100)
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(8, 48), lo=rng.randint(32, 96), hi=rng.randint(128, 400),
                    storage=rng.choice(["f32", "f32", "f16"]), steps=100 * rng.randint(5, 15))
    if kind == "serve":
        return dict(kind="serve", count=rng.randint(6, 24), lo=32, hi=rng.randint(64, 160), storage="f32",
                    steps=100 * rng.randint(4, 10))
    if kind == "scalar":
        nx = _log_int(rng, 128, 4096)
        ny = _log_int(rng, 128, 4096)
        budget = 2e8 if storage == "f64" else 8e9
        return dict(kind="scalar", nx=nx, ny=ny, storage=storage, steps=max(50, min(1000, int(budget / (nx * ny)))))
    if kind == "box":
        nx, ny, nz = (_log_int(rng, 24, 256) for _ in range(3))
        budget = 6e7 if storage == "f64" else 1e9
        return dict(kind="box", nx=nx, ny=ny, nz=nz, storage=storage,
                    Ra=float("%.3g" % math.exp(rng.uniform(math.log(1e4), math.log(1e7)))),
                    steps=max(10, min(400, int(budget / (nx * ny * nz)))))
    return dict(kind="boxes", count=rng.randint(4, 12), lo=rng.randint(16, 32), hi=rng.randint(48, 112),
                storage=rng.choice(["f32", "f16"]), steps=100 * rng.randint(2, 4))


# ------------------------------------------------------------------------------------------------
# Inputs


def _noise(shape, amplitude, gen):
    return (torch.rand(shape, generator=gen, dtype=torch.float64, device="cuda") - 0.5) * (2 * amplitude)


def _problem2d(c, seed):
    """(parameters, rho, ux, uy, T as device tensors, Nusselt axis) of a single 2-D lattice."""
    nx, ny = c["nx"], c["ny"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.arange(nx, dtype=torch.float64, device="cuda")[None, :]
    y = torch.arange(ny, dtype=torch.float64, device="cuda")[:, None]
    phase = torch.rand(4, generator=gen, dtype=torch.float64, device="cuda") * (2 * math.pi)
    rho = torch.ones((ny, nx), dtype=torch.float64, device="cuda")
    rates = {} if "rates" not in c else dict(s_3=c["rates"], s_4=c["rates"], lambda2=c["rates"])
    st = STORAGE[c["storage"]]
    if c["kind"] == "vortex":
        kx, ky = 2 * math.pi / nx, 2 * math.pi / ny
        U = 0.03
        ux = -U * torch.cos(kx * x + phase[0]) * torch.sin(ky * y + phase[1]) + _noise((ny, nx), 1e-4, gen)
        uy = U * torch.sin(kx * x + phase[0]) * torch.cos(ky * y + phase[1]) + _noise((ny, nx), 1e-4, gen)
        T = 0.1 * torch.sin(kx * x + phase[2]) * torch.sin(ky * y + phase[3]) + _noise((ny, nx), 1e-4, gen)
        p = W.default_params(nu=0.02, kappa=0.02, storage=st, u_ref=U, dT_ref=0.1, **rates)
        return p, rho, ux, uy, T, 1
    uc = 0.1
    if c["kind"] == "cavity":
        # developed state: hot and cold sides, one roll, a seeded disturbance
        nu, alpha, gb = W.convection_params(float(nx), c["Ra"], 0.71, uc)
        s = (x + 0.5) / nx
        h = (y + 0.5) / ny
        px, py = torch.sin(math.pi * s), torch.sin(math.pi * h)
        amp = 0.3 * uc * (1 + 0.2 * torch.sin(phase[0]))
        ux = amp * px * px * torch.sin(2 * math.pi * h) * -0.5 + _noise((ny, nx), 1e-4, gen)
        uy = amp * torch.sin(2 * math.pi * s) * py * py * 0.5 + _noise((ny, nx), 1e-4, gen)
        T = 0.5 - s + 0.1 * px * torch.cos(math.pi * h) + _noise((ny, nx), 1e-3, gen)
        p = W.default_params(nu=nu, kappa=alpha, g_beta=gb, storage=st, T_wall=(0.5, -0.5, 0.0, 0.0), u_ref=uc, dT_ref=1.0,
                             wall=(W.WALL_DIRICHLET, W.WALL_DIRICHLET, W.WALL_ADIABATIC, W.WALL_ADIABATIC), **rates)
        return p, rho, ux, uy, T, 0
    # layer heated from below: conduction profile, rolls about two heights wide, a seeded disturbance
    wet = bool(c.get("wet"))
    H = float(ny - 1 if wet else ny)
    nu, alpha, gb = W.convection_params(H, c["Ra"], 0.71, uc)
    h = (y if wet else y + 0.5) / H
    m = max(1, round(nx / (2 * H)))
    k = 2 * math.pi * m / nx
    psi = 0.3 * uc
    ux = psi * torch.cos(k * x + phase[0]) * torch.sin(2 * math.pi * h) * 0.5 + _noise((ny, nx), 1e-4, gen)
    uy = psi * torch.sin(k * x + phase[0]) * torch.sin(math.pi * h) ** 2 + _noise((ny, nx), 1e-4, gen)
    T = 0.5 - h + 0.1 * torch.sin(k * x + phase[0]) * torch.sin(math.pi * h) + _noise((ny, nx), 1e-3, gen)
    rho = rho * W.hydrostatic_density(h, gb, 1.0, H)
    kind = W.WALL_WET if wet else W.WALL_DIRICHLET
    p = W.default_params(nu=nu, kappa=alpha, g_beta=gb, storage=st, wall=(W.WALL_PERIODIC, W.WALL_PERIODIC, kind, kind),
                         T_wall=(0.0, 0.0, 0.5, -0.5), u_ref=uc, dT_ref=1.0, **rates)
    return p, rho, ux, uy, T, 1


def _problem_scalar(c, seed):
    """(parameters, T, ux, uy) of the prescribed-velocity case: a layer between Dirichlet walls in a
    cellular flow, as host arrays."""
    nx, ny = c["nx"], c["ny"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.arange(nx, dtype=torch.float64, device="cuda")[None, :]
    h = (torch.arange(ny, dtype=torch.float64, device="cuda")[:, None] + 0.5) / ny
    phase = torch.rand(1, generator=gen, dtype=torch.float64, device="cuda") * (2 * math.pi)
    k = 2 * math.pi * max(1, round(nx / (2 * ny))) / nx
    ux = 0.1 * torch.cos(k * x + phase) * torch.sin(2 * math.pi * h)
    uy = 0.1 * torch.sin(k * x + phase) * torch.sin(math.pi * h) ** 2
    T = 0.5 - h + 0.2 * torch.sin(k * x + phase) * torch.sin(math.pi * h) + _noise((ny, nx), 1e-2, gen)
    p = W.default_params(nu=0.05, kappa=0.05, storage=STORAGE[c["storage"]], T_wall=(0.0, 0.0, 0.5, -0.5), dT_ref=1.0,
                         wall=(W.WALL_PERIODIC, W.WALL_PERIODIC, W.WALL_DIRICHLET, W.WALL_DIRICHLET))
    return p, T.cpu().numpy(), ux.cpu().numpy(), uy.cpu().numpy()


def _problem_box(nx, ny, nz, Ra, storage, seed):
    """A 3-D layer heated from below with rolls and a seeded disturbance, as a Problem3D."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.arange(nx, dtype=torch.float64, device="cuda")[None, None, :]
    y = torch.arange(ny, dtype=torch.float64, device="cuda")[None, :, None]
    h = (torch.arange(nz, dtype=torch.float64, device="cuda")[:, None, None] + 0.5) / nz
    sh = (nz, ny, nx)
    phase = torch.rand(2, generator=gen, dtype=torch.float64, device="cuda") * (2 * math.pi)
    uc = 0.1
    nu, alpha, gb = W.convection_params(float(nz), Ra, 0.71, uc)
    if nu > 0.1:
        uc *= 0.1 / nu
        nu, alpha, gb = W.convection_params(float(nz), Ra, 0.71, uc)
    a, b = 2 * math.pi / nx * x + phase[0], 2 * math.pi / ny * y + phase[1]
    psi = 0.3 * uc
    ux = psi * torch.cos(a) * torch.cos(b) * torch.sin(2 * math.pi * h) * 0.5 + _noise(sh, 1e-4, gen)
    uy = psi * torch.sin(a) * torch.sin(b) * torch.sin(2 * math.pi * h) * -0.5 + _noise(sh, 1e-4, gen)
    uz = psi * torch.sin(a) * torch.cos(b) * torch.sin(math.pi * h) ** 2 + _noise(sh, 1e-4, gen)
    T = 0.5 - h + 0.1 * torch.sin(a) * torch.cos(b) * torch.sin(math.pi * h) + _noise(sh, 1e-3, gen)
    rho = torch.ones(sh, dtype=torch.float64, device="cuda") * W.hydrostatic_density(h, gb, 1.0, float(nz))
    p = W.default_params3(nu=nu, kappa=alpha, g_beta=gb, storage=STORAGE[storage], u_ref=uc, dT_ref=1.0,
                          wall=(W.WALL_PERIODIC,) * 4 + (W.WALL_DIRICHLET,) * 2, T_wall=(0.0,) * 4 + (0.5, -0.5))
    f = [t.cpu().numpy() for t in (rho, ux, uy, uz, T)]
    return W.Problem3D("box_%dx%dx%d" % sh[::-1], nx, ny, nz, p, *f)


def _boxes(c, seed):
    # the study's extents are part of the case; the states come from the seed
    shapes = np.random.default_rng(c["count"])
    out = []
    for k in range(c["count"]):
        e = np.exp(shapes.uniform(math.log(c["lo"]), math.log(c["hi"]), 3)).round().astype(int)
        Ra = float(np.exp(shapes.uniform(math.log(1e4), math.log(1e6))))
        out.append(_problem_box(int(e[0]), int(e[1]), int(e[2]), Ra, c["storage"], seed * 131 + k))
    return out


def _cavities(c, seed):
    shapes = np.random.default_rng(c["count"])
    out = []
    for k in range(c["count"]):
        n = int(round(math.exp(shapes.uniform(math.log(c["lo"]), math.log(c["hi"])))))
        Ra = float(np.exp(shapes.uniform(math.log(1e4), math.log(1e6))))
        case = dict(kind="cavity", nx=n, ny=n, storage=c["storage"], Ra=Ra)
        p, rho, ux, uy, T, axis = _problem2d(case, seed * 131 + k)
        out.append(W.Problem("cavity_%d" % n, n, n, p, *(t.cpu().numpy() for t in (rho, ux, uy, T)), nu_axis=axis))
    return out


def _requests(c, seed):
    trace = W.request_trace(c["count"], seed=c["count"], lo=c["lo"], hi=c["hi"], Ra_range=(2.5e3, 1e5),
                            storage=STORAGE[c["storage"]])
    out = []
    rng = np.random.default_rng(seed)
    for _, prob in trace:  # the trace's mix of shapes and kinds, with this seed's initial temperatures
        prob.T = prob.T + rng.uniform(-1e-2, 1e-2, prob.T.shape)
        out.append(prob)
    return out


# ------------------------------------------------------------------------------------------------
# The calls


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind in ("vortex", "cavity", "layer"):
        p, rho, ux, uy, T, axis = _problem2d(case, seed)
        s["lat"] = clb.Lattice(case["nx"], case["ny"], p)
        s["lat"].init_fields_device(rho, ux, uy, T)
        s["axis"] = axis
        s["out"] = [torch.empty_like(rho) for _ in range(4)]
        torch.cuda.synchronize()
    elif kind == "batch":
        s["batch"] = clb.Batch(_cavities(case, seed))
    elif kind == "serve":
        s["requests"] = _requests(case, seed)
        s["server"] = clb.Server(2 << 30, 64, STORAGE[case["storage"]])
    elif kind == "scalar":
        p, T, ux, uy = _problem_scalar(case, seed)
        s["scalar"] = clb.Thermal(case["nx"], case["ny"], p)
        s["scalar"].init(T, ux, uy)
    elif kind == "box":
        prob = _problem_box(case["nx"], case["ny"], case["nz"], case["Ra"], case["storage"], seed)
        s["lat"] = clb.Lattice3D.from_problem(prob)
    else:
        s["batch"] = clb.Batch3D(_boxes(case, seed))
    return s


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind in ("vortex", "cavity", "layer"):
        lat = s["lat"]
        out = {}
        if c["every"]:
            # run() without a tolerance that the run can meet: all steps, a residual check every `every`
            out["steps"], out["residual"] = lat.run(0.0, c["steps"], c["every"])
            out["nusselt"] = lat.nusselt(s["axis"])
        else:
            lat.step(c["steps"])
        lat.fields_device(*s["out"])
        out["fields"] = s["out"]
        return out
    if kind == "batch":
        b = s["batch"]
        b.step(c["steps"])
        nu, er = b.diagnostics()
        fields = [b.fields(k) for k in range(len(b))]
        return {"nusselt": nu, "residual": er, "fields": [np.concatenate([f[q].ravel() for f in fields]) for q in range(4)]}
    if kind == "serve":
        srv = s["server"]
        ids = [srv.submit(r, step_cap=c["steps"], tol=0.0) for r in s["requests"]]
        while True:
            active, queued = srv.progress(100)
            if not active and not queued:
                break
        polled = [srv.poll(i) for i in ids]
        fields = [srv.fetch(i, r.ny, r.nx) for i, r in zip(ids, s["requests"])]
        return {"nusselt": np.array([p[1] for p in polled]), "steps": np.array([p[2] for p in polled]),
                "residual": np.array([p[3] for p in polled]),
                "fields": [np.concatenate([f[q].ravel() for f in fields]) for q in range(4)]}
    if kind == "scalar":
        s["scalar"].step(c["steps"])
        return {"fields": [s["scalar"].temperature()]}
    if kind == "box":
        s["lat"].step(c["steps"])
        return {"nusselt": s["lat"].nusselt(2), "fields": list(s["lat"].fields())}
    b = s["batch"]
    b.step(c["steps"])
    fields = [b.fields(k) for k in range(len(b.problems))]
    return {"fields": [np.concatenate([f[q].ravel() for f in fields]) for q in range(5)]}


def _nodes(case):
    if case["kind"] == "batch":
        shapes = np.random.default_rng(case["count"])
        n = 0
        for _ in range(case["count"]):
            n += int(round(math.exp(shapes.uniform(math.log(case["lo"]), math.log(case["hi"]))))) ** 2
            shapes.uniform()
        return n
    if case["kind"] == "serve":
        return sum(p.nodes for p in _requests(case, 0))
    if case["kind"] == "boxes":
        shapes = np.random.default_rng(case["count"])
        n = 0
        for _ in range(case["count"]):
            n += int(np.prod(np.exp(shapes.uniform(math.log(case["lo"]), math.log(case["hi"]), 3)).round()))
            shapes.uniform()
        return n
    return case["nx"] * case["ny"] * case.get("nz", 1)


def work(case):
    """The populations (and a prescribed velocity) read once and written once per pass, the fields
    written once; the arithmetic of every node update."""
    pops, fields, flops = {"scalar": (5, 1, 45), "box": (34, 5, 550), "boxes": (34, 5, 550)}.get(case["kind"], (14, 4, 209))
    n = _nodes(case)
    e = BYTES[case["storage"]]
    bytes_ = n * (2 * pops * e + 8 * fields)
    if case["kind"] == "scalar":
        bytes_ += n * 2 * max(e, 4)
    return {"bytes": float(bytes_), "flops": float(n) * case["steps"] * flops}


# ------------------------------------------------------------------------------------------------
# The same initial state advanced in FP64 with plain torch operations


class _Exact:
    """The coupled (or temperature-only) method on one lattice of d = 2 or 3 axes. Arrays run over
    (velocity, [z,] y, x); tensors of velocity digits run over x fastest, digit 0, 1, 2 standing for
    e = 0, +1, -1. Walls: periodic, Dirichlet and adiabatic (half-way), and in 2-D the paper's own
    conditions on the y sides."""

    def __init__(self, p, shape):
        self.p, self.d, self.shape = p, len(shape), shape  # shape: ([nz,] ny, nx)
        d = self.d
        one = torch.tensor([[1.0, 1, 1], [0, 1, -1], [0, 1, 1]], dtype=torch.float64)
        inv = torch.linalg.inv(one)
        M, I = one, inv
        for _ in range(d - 1):
            M, I = torch.kron(one, M), torch.kron(inv, I)
        self.M, self.I = M.cuda(), I.cuda()
        self.digits = [tuple(reversed(t)) for t in itertools.product(range(3), repeat=d)]  # x fastest
        v = (0, 1, -1)
        self.e = [tuple(v[a] for a in t) for t in self.digits]
        self.opp = [self.digits.index(tuple((0, 2, 1)[a] for a in t)) for t in self.digits]
        self.ge = [tuple([0] * d)] + [tuple(s if a == b else 0 for b in range(d)) for a in range(d) for s in (1, -1)]
        self.s_nu = 1.0 / (3.0 * p["nu"] + 0.5)
        self.l1 = 1.0 / (p["kappa"] / p["cs2_T"] + 0.5)
        self.gravity = p.get("g_axis", 1)

    def axis(self, a):  # the array dimension of axis a (after the velocity dimension)
        return self.d - a

    def lin(self, A, f):
        return (A @ f.reshape(f.shape[0], -1)).reshape(f.shape)

    def shift(self, m, u, sign):
        """Moments about 0 to moments about u (sign = -1), or back (sign = +1), axis by axis."""
        for a in range(self.d):
            step = 3 ** a
            for k, t in enumerate(self.digits):
                if t[a] == 0:
                    w = sign * u[a]
                    m[k + 2 * step] += w * (2 * m[k + step] + w * m[k])
                    m[k + step] += w * m[k]
        return m

    def maxwell(self):
        return [math.prod((1.0, 0.0, 1.0 / 3.0)[a] for a in t) for t in self.digits]

    def equilibrium(self, rho, u):
        k = torch.stack([rho * c for c in self.maxwell()])
        return self.lin(self.I, self.shift(k, u, 1))

    def g_equilibrium(self, T, u):
        return self.g_back(T, [torch.zeros_like(T)] * self.d, [self.p["cs2_T"] * T] * self.d, u)

    def g_back(self, T, k1, k2, u):
        out, rest = [None], T
        for a in range(self.d):
            r1 = k1[a] + u[a] * T
            r2 = k2[a] + 2 * u[a] * k1[a] + u[a] * u[a] * T
            rest = rest - r2
            out += [0.5 * (r2 + r1), 0.5 * (r2 - r1)]
        out[0] = rest
        return torch.stack(out)

    def init(self, rho, u, T):
        self.f = self.equilibrium(rho, u)
        self.g = self.g_equilibrium(T, u)

    def macro(self, f, g):
        T = g.sum(0)
        rho = f.sum(0)
        F = [torch.full_like(T, self.p["Fv"][a]) for a in range(self.d)]
        F[self.gravity] = F[self.gravity] + self.p["rho0"] * self.p["g_beta"] * (T - self.p["T0"])
        u = []
        for a in range(self.d):
            j = sum(f[k] if e[a] > 0 else -f[k] for k, e in enumerate(self.e) if e[a])
            u.append((j + 0.5 * F[a]) / rho)
        return rho, u, T, F

    def collide_f(self, f, rho, u, F):
        p, d = self.p, self.d
        m = self.shift(self.lin(self.M, f), u, -1)
        a = [m[2 * 3 ** b] - rho / 3 for b in range(d)]
        trace = (p["s_b"] - self.s_nu) / d * sum(a)
        rate = {2: self.s_nu, 3: p["s_3"], 4: p["s_4"], 5: p.get("s_5"), 6: p.get("s_6")}
        for k, (t, c) in enumerate(zip(self.digits, self.maxwell())):
            order = sum(t)
            ones = [b for b in range(d) if t[b] == 1]
            if order == 0:
                continue
            if order == 1:
                m[k] += F[ones[0]]
            elif order == 2 and not ones:
                b = t.index(2)
                m[k] -= self.s_nu * a[b] + trace
            else:
                s = rate[order]
                m[k] -= s * (m[k] - c * rho)
                if len(ones) == 1:
                    m[k] += (1 - 0.5 * s) * math.prod(1.0 / 3.0 for b in t if b == 2) * F[ones[0]]
        return self.lin(self.I, self.shift(m, u, 1))

    def collide_g(self, g, u, T):
        k1, k2 = [], []
        for a in range(self.d):
            gp, gm = g[1 + 2 * a], g[2 + 2 * a]
            c1 = gp - gm - u[a] * T
            c2 = gp + gm - 2 * u[a] * (gp - gm) + u[a] * u[a] * T
            k1.append((1 - self.l1) * c1)
            k2.append(c2 - self.p["lambda2"] * (c2 - self.p["cs2_T"] * T))
        return self.g_back(T, k1, k2, u)

    def stream(self, f, es, opps, temperature):
        p = self.p
        out = torch.empty_like(f)
        for k, e in enumerate(es):
            r = torch.roll(f[k], [e[a] for a in range(self.d)], [self.d - 1 - a for a in range(self.d)])
            for a in range(self.d):
                face = 2 * a + (0 if e[a] > 0 else 1)
                if e[a] and p["wall"][face] != W.WALL_PERIODIC:
                    edge = 0 if e[a] > 0 else self.shape[self.d - 1 - a] - 1
                    back = f[opps[k]].select(self.d - 1 - a, edge)
                    if temperature and p["wall"][face] == W.WALL_DIRICHLET:
                        back = p["cs2_T"] * p["T_wall"][face] - back
                    r.select(self.d - 1 - a, edge).copy_(back)
            out[k] = r
        return out

    def wet_rows(self):
        """The paper's conditions on the end rows of a 2-D layer (both y sides, periodic x)."""
        p = self.p
        f, g = self.f, self.g
        for face, row, inner, n in ((2, 0, 1, 1), (3, self.shape[0] - 1, self.shape[0] - 2, -1)):
            Tw = p["T_wall"][face]
            fq, gq = f[:, inner:inner + 1], g[:, inner:inner + 1]
            _, uq, Tq, _ = self.macro(fq, gq)
            fw = f[:, row]
            Fy = p["Fv"][1] + p["rho0"] * p["g_beta"] * (Tw - p["T0"])
            Fx = p["Fv"][0]
            Z = sum(fw[k] for k, e in enumerate(self.e) if e[1] == 0)
            O = sum(fw[k] for k, e in enumerate(self.e) if e[1] == -n)
            rho = Z + 2 * O - 0.5 * n * Fy
            u = [-0.5 * Fx / rho, -0.5 * Fy / rho]
            feq = self.equilibrium(rho, u)
            for k, e in enumerate(self.e):
                if e[1] == n:
                    fw[k] = fw[self.opp[k]] + feq[k] - feq[self.opp[k]]
            St = sum(e[0] * fw[k] for k, e in enumerate(self.e) if e[0])
            delta = 0.5 * (rho * u[0] - St)
            for k, e in enumerate(self.e):
                if e[1] == n and e[0]:
                    fw[k] += e[0] * delta
            zero = torch.zeros_like(rho)
            ge_w = self.g_equilibrium(torch.full_like(rho, Tw), [zero, zero])
            ge_q = self.g_equilibrium(Tq[0], [v[0] for v in uq])
            g[:, row] = ge_w + gq[:, 0] - ge_q

    def step(self):
        rho, u, T, F = self.macro(self.f, self.g)
        f, g = self.collide_f(self.f, rho, u, F), self.collide_g(self.g, u, T)
        self.f = self.stream(f, self.e, self.opp, False)
        self.g = self.stream(g, self.ge, [0] + [1 + (j ^ 1) for j in range(2 * self.d)], True)
        if self.p["wall"][2] == W.WALL_WET:
            self.wet_rows()

    def scalar_step(self, u):
        g = self.collide_g(self.g, u, self.g.sum(0))
        self.g = self.stream(g, self.ge, [0] + [1 + (j ^ 1) for j in range(2 * self.d)], True)


def _exact_nusselt(p, rho, u, T, axis):
    lo, hi = p["T_wall"][2 * axis], p["T_wall"][2 * axis + 1]
    dT = abs(lo - hi) or 1.0
    q = u[axis] * (T - p["T0"])
    n = list(reversed(T.shape))
    cells, H = float(math.prod(n)), n[axis]
    if p["wall"][2] == W.WALL_WET:  # walls on the end rows: the trapezoid rule
        q = torch.cat([0.5 * q[:1], q[1:-1], 0.5 * q[-1:]])
        cells, H = float(n[0] * (n[1] - 1)), n[axis] - (1 if axis == 1 else 0)
    return 1.0 + (1.0 if lo >= hi else -1.0) * float(q.sum()) / cells * H / (p["kappa"] * dT)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        return None
    three = kind in ("box", "boxes")
    if _nodes(case) * case["steps"] > (EXACT_LIMIT_3D if three else EXACT_LIMIT_2D):
        return None
    if kind == "boxes":
        probs = _boxes(case, seed)
        if sum(case["steps"] for _ in probs) > 6000:
            return None
        got = []
        for prob in probs:
            E = _Exact(prob.params, prob.shape)
            rho, ux, uy, uz, T = (torch.from_numpy(a).cuda() for a in prob.fields())
            E.init(rho, [ux, uy, uz], T)
            for _ in range(case["steps"]):
                E.step()
            rho, u, T, _ = E.macro(E.f, E.g)
            got.append([rho, *u, T])
        return {"fields": [torch.cat([f[q].reshape(-1) for f in got]).cpu().numpy() for q in range(5)]}
    if kind == "box":
        prob = _problem_box(case["nx"], case["ny"], case["nz"], case["Ra"], case["storage"], seed)
        E = _Exact(prob.params, prob.shape)
        rho, ux, uy, uz, T = (torch.from_numpy(a).cuda() for a in prob.fields())
        E.init(rho, [ux, uy, uz], T)
        for _ in range(case["steps"]):
            E.step()
        rho, u, T, _ = E.macro(E.f, E.g)
        return {"nusselt": _exact_nusselt(prob.params, rho, u, T, 2), "fields": [rho, *u, T]}
    if kind == "scalar":
        p, T, ux, uy = _problem_scalar(case, seed)
        T, ux, uy = (torch.from_numpy(a).cuda() for a in (T, ux, uy))
        E = _Exact(p, tuple(T.shape))
        E.g = E.g_equilibrium(T, [ux, uy])
        for _ in range(case["steps"]):
            E.scalar_step([ux, uy])
        return {"fields": [E.g.sum(0)]}
    p, rho, ux, uy, T, axis = _problem2d(case, seed)
    E = _Exact(p, tuple(T.shape))
    E.init(rho, [ux, uy], T)
    if p["wall"][2] == W.WALL_WET:
        E.wet_rows()  # the conditions hold from the start
    for _ in range(case["steps"]):
        E.step()
    rho, u, T, _ = E.macro(E.f, E.g)
    out = {"fields": [rho, u[0], u[1], T]}
    if case["every"]:
        # the steps and the residual against the snapshot of the last check have no value here
        out.update(steps=None, residual=None, nusselt=_exact_nusselt(p, rho, u, T, axis))
    return out
