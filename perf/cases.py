"""What a user of the lattice Boltzmann library has it do, as cases to measure.

A case is a run through the public Python binding: a lattice (nozzle, pipe or
periodic vortex) advanced by a number of time steps with its result read back,
a restart from given populations, or a stream of requests through the server.
Results go to the GPU as PyTorch tensors in the lattice's storage precision
(FP64, FP32, or FP32 density and FP16 velocity for FP16S), which is how a
PyTorch program that post-processes the flow takes them.

exact() advances the same inputs in plain PyTorch, in 64 bits, from the
definitions of the method: pull streaming with halfway or interpolated
bounce-back, central Hermite moments relaxed order by order, and the
non-equilibrium-extrapolation inlet and outlet.
"""
import functools
import math

import numpy as np
import torch

from paper_2204_10566_gb300 import inputs as I
from paper_2204_10566_gb300 import lbm, serving

U_THROAT = 0.05      # throat mean velocity of the nozzle and pipe runs (lattice units)
VORTEX_U0 = 0.04     # velocity amplitude of the Taylor-Green vortex
STORAGE = {"fp64": 8, "fp32": 4, "fp16s": 2}
# floating-point operations per cell update: the rate-1 collision, and the full 27-moment cascade
FLOPS_RATE1, FLOPS_CASCADE = 400, 800


# ------------------------------------------------------------------- cases

def _pipe_or_nozzle(kind, D, d, length, precision, steps, re, profile="parabolic", noise=0.01, ramp=8000,
                    walls="halfway", stats="none"):
    return dict(kind=kind, D=D, d=d, length=length, precision=precision, steps=steps, re=re, profile=profile,
                noise=noise, ramp=ramp, walls=walls, stats=stats)


def listed():
    def case(name, c):
        return dict(c, name=name)

    P = _pipe_or_nozzle
    return [
        # the laminar Re 500 nozzle at its own 200 steps: a lattice that fits L2, launches and latency count
        case("laminar_nozzle_fp32", P("nozzle", 24, 8, 160, "fp32", 200, 500.0, "plug", 0.0, 0)),
        # one pipe request of the serving range run on its own: odd, small sizes, half-precision storage
        case("small_pipe_fp16s", P("pipe", 33, 11, 275, "fp16s", 100, 2000.0, ramp=25)),
        # restart of the laminar nozzle from host populations, a few steps, populations back to the host
        case("restart_fp32", dict(kind="restart", D=24, d=8, length=160, precision="fp32", steps=40, re=500.0)),
        # the transitional Re 3500 nozzle between two readouts of the flow
        case("nozzle_re3500_fp32", P("nozzle", 96, 32, 800, "fp32", 200, 3500.0)),
        # the same run while it averages the axial velocity and its square on every step
        case("nozzle_re3500_averages_fp32", P("nozzle", 96, 32, 800, "fp32", 100, 3500.0, stats="axial")),
        # the same nozzle with the smooth-surface walls of the paper (interpolated bounce-back)
        case("nozzle_re3500_smooth_fp32", P("nozzle", 96, 32, 800, "fp32", 200, 3500.0, walls="smooth")),
        # the FP64 run that the reduced storage precisions are compared with
        case("nozzle_re3500_fp64", P("nozzle", 96, 32, 800, "fp64", 25, 3500.0)),
        # the under-resolved Re 6500 nozzle, the largest grid, in both production precisions
        case("nozzle_re6500_fp32", P("nozzle", 144, 48, 1200, "fp32", 200, 6500.0, noise=0.02)),
        case("nozzle_re6500_fp16s", P("nozzle", 144, 48, 1200, "fp16s", 200, 6500.0, noise=0.02)),
        # one point of a Reynolds sweep on the periodic vortex: upload, run, read back
        case("vortex_256_fp32", dict(kind="vortex", n=256, precision="fp32", steps=100, re=1600.0, ghost="one")),
        # the ghost-rate study: every order relaxed at omega (lattice BGK), the general collision
        case("vortex_64_bgk_fp32", dict(kind="vortex", n=64, precision="fp32", steps=200, re=1600.0, ghost="omega")),
        # a burst of mixed nozzle and pipe requests through the server, until every result is back
        case("serving_mix", dict(kind="serving", requests=12, mix=2204, d_min=8, d_max=16, steps_min=300,
                                 steps_max=900, steps_per_tick=32)),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["nozzle", "nozzle", "pipe", "pipe", "vortex", "restart", "serving"])
    if kind == "serving":
        lo = rng.randint(6, 10)
        return dict(kind=kind, requests=rng.randint(4, 14), mix=rng.randint(1, 10 ** 6), d_min=lo,
                    d_max=lo + rng.randint(2, 6), steps_min=rng.randint(200, 400), steps_max=rng.randint(500, 900),
                    steps_per_tick=rng.choice([16, 32, 64]))
    if kind == "restart":
        d = rng.randint(5, 14)
        return dict(kind=kind, D=3 * d + rng.randint(0, 1), d=d, length=rng.randint(15 * d, 25 * d),
                    precision=rng.choice(["fp32", "fp64"]), steps=rng.randint(10, 100), re=float(rng.randint(500, 2000)))
    if kind == "vortex":
        c = dict(kind=kind, n=_log(rng, 24, 256), precision=rng.choice(["fp32", "fp32", "fp16s", "fp64"]),
                 steps=_log(rng, 20, 400), re=float(rng.choice([100, 400, 1600])),
                 ghost=rng.choice(["one", "one", "omega"]))
    else:
        d = _log(rng, 5, 48)
        D = 3 * d + rng.randint(0, 1)
        c = _pipe_or_nozzle(kind, D, d, rng.randint(15 * d, 25 * d), rng.choice(["fp32", "fp32", "fp16s", "fp64"]),
                            _log(rng, 20, 400), float(rng.randint(500, 6500)), rng.choice(["plug", "parabolic"]),
                            rng.choice([0.0, 0.01, 0.02]), 8000, rng.choice(["halfway", "halfway", "smooth"]),
                            rng.choice(["none", "none", "none", "axial", "full"]))
    # no more cell updates than the largest listed case, FP64, the general collision and averages weighed by their cost
    weight = {"fp64": 20, "fp32": 1, "fp16s": 1}[c["precision"]] * (3 if c.get("ghost") == "omega" else 1)
    weight *= {"none": 1, "axial": 2, "full": 5}[c.get("stats", "none")] * (2 if c.get("walls") == "smooth" else 1)
    box = c["n"] ** 3 if kind == "vortex" else 0.8 * c["D"] ** 2 * c["length"]
    c["steps"] = max(1, min(c["steps"], int(2.0e9 / (box * weight))))
    return c


# ------------------------------------------------------------------ inputs

@functools.lru_cache(maxsize=4)
def _flags(kind, D, d, length):
    return I.pipe_flags(D, length) if kind == "pipe" else I.nozzle_flags(D, d, length)


@functools.lru_cache(maxsize=2)
def _wall_q(kind, D, d, length):
    flags = _flags(kind, D, d, length)
    if kind == "pipe":
        return I.nozzle_wall_q(D, D, length, L_in=length, L_cone=1, L_throat=0, flags=flags)
    return I.nozzle_wall_q(D, d, length, flags=flags)


def _params(case, seed):
    """The flow parameters of a nozzle, pipe or restart case."""
    return dict(Re=case["re"], u_char=U_THROAT, L_char=float(case["d"]), u_in=U_THROAT * (case["d"] / case["D"]) ** 2,
                d_in=float(case["D"]), profile=case.get("profile", "plug"), noise_amp=case.get("noise", 0.0),
                noise_seed=int(seed), inlet_ramp=case.get("ramp", 0))


def _vortex_nu(case):
    return VORTEX_U0 * case["n"] / (2 * math.pi) / case["re"]


def _omega(nu):
    return 1.0 / (3.0 * nu + 0.5)


def _ghost(case):
    return ((_omega(_vortex_nu(case)),) if case.get("ghost") == "omega" else (1.0,)) * 4


def _random(shape, seed):
    """Uniform numbers in [-1, 1), in 64 bits, on the host."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    g = torch.Generator(dev).manual_seed(int(seed))
    return (2.0 * torch.rand(shape, generator=g, device=dev, dtype=torch.float64) - 1.0).cpu().numpy()


def _fields(case, n, seed):
    """Initial density and velocity of the n active cells: small random
    fluctuations about the state at rest (nozzle and pipe), or the
    Taylor-Green vortex at a random position of its box."""
    if case["kind"] != "vortex":
        r = _random((4 * n,), seed)
        return 1.0 + 0.001 * r[:n], 0.01 * r[n:].reshape(n, 3)
    k = 2 * np.pi / case["n"]
    shift = np.random.default_rng(seed).uniform(0.0, 2 * np.pi, 3)
    c = k * (np.arange(case["n"]) + 0.5)
    x, y, z = (c + shift[0])[None, None, :], (c + shift[1])[None, :, None], (c + shift[2])[:, None, None]
    u = np.zeros((case["n"],) * 3 + (3,))
    u[..., 0] = VORTEX_U0 * np.sin(x) * np.cos(y) * np.cos(z)
    u[..., 1] = -VORTEX_U0 * np.cos(x) * np.sin(y) * np.cos(z)
    p = VORTEX_U0 ** 2 / 16.0 * (np.cos(2 * x) + np.cos(2 * y)) * (np.cos(2 * z) + 2.0)
    return (1.0 + 3.0 * p).reshape(-1), u.reshape(-1, 3)


def _velocities():
    return np.array([[i % 3 - 1, (i // 3) % 3 - 1, i // 9 - 1] for i in range(27)], dtype=np.float64)


def _weights():
    w1 = np.array([1.0 / 6.0, 2.0 / 3.0, 1.0 / 6.0])
    return np.array([w1[i % 3] * w1[(i // 3) % 3] * w1[i // 9] for i in range(27)])


def _populations(case, n, seed):
    """Saved populations to restart from: near equilibrium, with a random non-equilibrium part."""
    r = _random((n, 31), seed)
    rho, u = 1.0 + 0.001 * r[:, 27:28], 0.01 * r[:, 28:]
    cu = u @ _velocities().T
    feq = rho * _weights() * (1.0 + 3.0 * cu + 4.5 * cu ** 2 - 1.5 * (u ** 2).sum(1, keepdims=True))
    return feq * (1.0 + 0.001 * r[:, :27])


def _requests(case, seed):
    """(flags, steps, precision, parameters) of each request of a serving case."""
    specs = I.serving_requests(case["requests"], seed=case["mix"], d_range=(case["d_min"], case["d_max"]),
                               steps_range=(case["steps_min"], case["steps_max"]))
    out = []
    for s in specs:
        p = serving.request_params(s)
        p["noise_seed"] = int(seed) * 64 + s["id"]
        out.append((serving.request_geometry(s), s["steps"], s["precision"], p))
    return out


# --------------------------------------------------------------- the passes

def _pinned(n):
    """Page-locked host arrays for the moments of n cells."""
    return (torch.empty(n, dtype=torch.float64, pin_memory=True).numpy(),
            torch.empty((n, 3), dtype=torch.float64, pin_memory=True).numpy())


def prepare(case, seed):
    if case["kind"] == "serving":
        return dict(case=case, server=lbm.Server(16 << 30, max_slots=32, steps_per_tick=case["steps_per_tick"]),
                    requests=_requests(case, seed))
    if case["kind"] == "vortex":
        n = case["n"]
        lat = lbm.Lattice(I.box_flags(n, n, n), case["precision"], periodic=7)
        lat.set_params(nu=_vortex_nu(case), ghost=_ghost(case))
        fields = tuple(torch.from_numpy(a).pin_memory().numpy() for a in _fields(case, lat.n_active, seed))
        return dict(case=case, lattice=lat, fields=fields, out=_pinned(lat.n_active))
    geometry = (case["kind"], case["D"], case["d"], case["length"])
    lat = lbm.Lattice(_flags(*geometry), case["precision"])
    lat.set_params(**_params(case, seed))
    if case["kind"] == "restart":
        return dict(case=case, lattice=lat, populations=_populations(case, lat.n_active, seed))
    if case["walls"] == "smooth":
        lat.set_wall_q(*_wall_q(*geometry))
    lat.init_fields(*_fields(case, lat.n_active, seed))
    if case["stats"] != "none":
        lat.stats_begin(1, full=case["stats"] == "full")
    return dict(case=case, lattice=lat, out=_pinned(lat.n_active))


def _to_gpu(a, dtype):
    return torch.from_numpy(a).to("cuda").to(dtype)


def _moments(rho, u, precision):
    rho_type = torch.float64 if precision == "fp64" else torch.float32
    u_type = torch.float16 if precision == "fp16s" else rho_type
    return [_to_gpu(rho, rho_type), _to_gpu(u, u_type)]


def run(state):
    case = state["case"]
    if case["kind"] == "serving":
        srv = state["server"]
        ids = [srv.submit(flags, steps, precision, **p) for flags, steps, precision, p in state["requests"]]
        done = {}
        while len(done) < len(ids):
            srv.tick()
            for k, rid in enumerate(ids):
                if k not in done and srv.poll(rid)[0] in (lbm.LBM_REQ_DONE, lbm.LBM_REQ_FAILED):
                    done[k] = _moments(*srv.result(rid), state["requests"][k][2])
        return [done[k] for k in range(len(ids))]
    lat, precision = state["lattice"], case["precision"]
    if case["kind"] == "restart":
        lat.set_populations(state["populations"])
        lat.step(case["steps"])
        return _to_gpu(lat.get_populations(), torch.float64 if precision == "fp64" else torch.float32)
    if case["kind"] == "vortex":
        lat.init_fields(*state["fields"])
    lat.step(case["steps"])
    out = _moments(*lat.moments(out=state["out"]), precision)
    real = torch.float64 if precision == "fp64" else torch.float32
    if case.get("stats") == "axial":
        out += [_to_gpu(m, real) for m in lat.stats_get()[:2]]
    elif case.get("stats") == "full":
        means = lat.stats_get_full()
        out += [_to_gpu(np.ascontiguousarray(means[k]), real) for k in ("u", "uu", "sigma", "rho")]
    return out


# -------------------------------------------------------------------- work

def _cells(case):
    if case["kind"] == "vortex":
        return case["n"] ** 3
    return I.active_count(_flags(case["kind"], case["D"], case["d"], case["length"]))


def work(case):
    """One pass: every step reads and writes 27 populations of each cell once
    in the storage precision (and the accumulators of the averages), plus the
    fields that cross the public interface."""
    if case["kind"] == "serving":
        updates = bytes_ = results = 0
        for flags, steps, precision, _ in _requests(case, 0):
            n = I.active_count(flags)
            updates += n * steps
            bytes_ += n * steps * 54 * STORAGE[precision]
            results += flags.size + n * 32
        return {"bytes": bytes_ + results, "flops": updates * FLOPS_RATE1}
    n, s = _cells(case), STORAGE[case["precision"]]
    averages = {"none": 0, "axial": 2, "full": 18}[case.get("stats", "none")]
    step = 54 * s + averages * 16
    io = 2 * 27 * 8 if case["kind"] == "restart" else 32 + (32 if case["kind"] == "vortex" else 0)
    io += {0: 0, 2: 16, 18: 128}[averages]
    flops = FLOPS_CASCADE if case.get("ghost") == "omega" else FLOPS_RATE1
    return {"bytes": n * (case["steps"] * step + io), "flops": n * case["steps"] * flops}


# ------------------------------------------------------------------- exact

class _Plain:
    """The method in plain PyTorch, in 64 bits: populations f[27][n] of the
    active cells in increasing box order."""

    CHUNK = 1 << 21

    def __init__(self, flags, periodic, omega, ghost=(1.0,) * 4, params=None, wall_q=None):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        dev = self.dev
        self.flags = torch.from_numpy(np.ascontiguousarray(flags)).to(dev)
        nz, ny, nx = self.flags.shape
        self.size = (nx, ny, nz)
        act = torch.nonzero(self.flags.reshape(-1)).reshape(-1)
        self.n = n = act.numel()
        self.box = act
        index = torch.full((flags.size,), -1, dtype=torch.int32, device=dev)
        index[act] = torch.arange(n, dtype=torch.int32, device=dev)
        x, y, z = act % nx, (act // nx) % ny, act // (nx * ny)
        self.kind = self.flags.reshape(-1)[act]
        self.c = [[i % 3 - 1, (i // 3) % 3 - 1, i // 9 - 1] for i in range(27)]
        self.w = torch.from_numpy(_weights()).to(dev)[:, None]
        self.index = index

        def neighbour(cx, cy, cz):
            """Active index of the cell at x - c, or -1 for a wall."""
            p = [x - cx, y - cy, z - cz]
            inside = torch.ones(n, dtype=torch.bool, device=dev)
            for a in range(3):
                if periodic:
                    p[a] = p[a] % self.size[a]
                else:
                    inside &= (p[a] >= 0) & (p[a] < self.size[a])
                    p[a] = p[a].clamp(0, self.size[a] - 1)
            return torch.where(inside, index[p[0] + nx * (p[1] + ny * p[2])], -1)

        me = torch.arange(n, dtype=torch.int32, device=dev)
        self.src = torch.empty((27, n), dtype=torch.int32, device=dev)
        walls = []
        for i in range(27):
            s = neighbour(*self.c[i])
            walls.append(s < 0)
            self.src[i] = torch.where(s >= 0, s + i * n, me + (26 - i) * n)
        # interpolated bounce-back: cells, whether each link and its opposite end at a wall, distances
        self.q = None
        if wall_q is not None:
            cells = index[torch.from_numpy(wall_q[0]).to(dev)].long()
            q = torch.from_numpy(wall_q[1]).to(dev).double().T / 256.0
            self.q = (cells, torch.stack([walls[i][cells] for i in range(27)]), q)
        # inlet and outlet nodes: the unique axis neighbour that is a fluid cell
        self.nodes = torch.nonzero(self.kind >= 2).reshape(-1)
        if self.nodes.numel():
            k = self.nodes
            self.partner = torch.full_like(k, -1)
            self.normal = torch.zeros((3, k.numel()), dtype=torch.float64, device=dev)
            for a in range(3):
                for s in (1, -1):
                    c = [0, 0, 0]
                    c[a] = -s
                    j = neighbour(*c)[k].long()
                    fluid = (j >= 0) & (self.kind[j.clamp(min=0)] == 1)
                    self.partner = torch.where(fluid, j, self.partner)
                    self.normal[a][fluid] = float(s)
        self.omega, self.rates, self.p = omega, (omega,) + tuple(ghost), params
        self.xy = (x[self.nodes].double() + 0.5 - nx / 2.0, y[self.nodes].double() + 0.5 - ny / 2.0)
        self.t = 0

    @staticmethod
    def _axis(u):
        """1-D equilibrium factors and inverse columns g0, g1, g2 at c = -1, 0, 1."""
        g0 = [1.0 / 6.0 + 0.5 * (u * u - u), 2.0 / 3.0 - u * u, 1.0 / 6.0 + 0.5 * (u * u + u)]
        return g0, [u - 0.5, -2.0 * u, u + 0.5], [0.5, -1.0, 0.5]

    def equilibrium(self, rho, u):
        X, Y, Z = (self._axis(u[a])[0] for a in range(3))
        return torch.stack([rho * X[i % 3] * Y[(i // 3) % 3] * Z[i // 9] for i in range(27)])

    def start(self, rho, u):
        rho, u = torch.from_numpy(np.ascontiguousarray(rho)).to(self.dev), torch.from_numpy(np.ascontiguousarray(u.T)).to(self.dev)
        self.f = torch.empty((27, self.n), dtype=torch.float64, device=self.dev)
        for b in range(0, self.n, self.CHUNK):
            e = slice(b, b + self.CHUNK)
            self.f[:, e] = self.equilibrium(rho[e], u[:, e])
        return self

    def moments(self, f):
        rho = f.sum(0)
        j = [sum(float(c[a]) * f[i] for i, c in enumerate(self.c) if c[a]) for a in range(3)]
        return rho, torch.stack(j) / rho

    def collide(self, f, rho, u):
        """T^-1 S T (f^eq - f) + f, and the second-order central Hermite moments."""
        m = f.reshape(3, 3, 3, -1)  # [z][y][x]
        for axis, a in ((2, 0), (1, 1), (0, 2)):
            lo, mid, hi = m.unbind(axis)
            s, d = lo + hi, hi - lo
            m0 = s + mid
            m = torch.stack([m0, d - u[a] * m0, s - 2.0 * u[a] * d + (u[a] * u[a] - 1.0 / 3.0) * m0], axis)
        second = torch.stack([m[0, 0, 2], m[0, 2, 0], m[2, 0, 0], m[0, 1, 1], m[1, 0, 1], m[1, 1, 0]])
        keep = torch.empty((3, 3, 3, 1), dtype=torch.float64, device=self.dev)
        for kz in range(3):
            for ky in range(3):
                for kx in range(3):
                    order = kx + ky + kz
                    keep[kz, ky, kx] = 0.0 if order < 2 else 1.0 - self.rates[order - 2]
        m = m * keep
        m[0, 0, 0] = rho
        for axis, a in ((0, 2), (1, 1), (2, 0)):
            m0, m1, m2 = m.unbind(axis)
            g0, g1, g2 = self._axis(u[a])
            m = torch.stack([g0[c] * m0 + g1[c] * m1 + g2[c] * m2 for c in range(3)], axis)
        return m.reshape(27, -1), second

    def _inlet(self, rho_f, u_f):
        """Density and velocity prescribed at the inlet and outlet nodes."""
        p, inlet = self.p, self.kind[self.nodes] == 2
        speed = torch.full_like(rho_f, p["u_in"])
        if p["profile"] == "parabolic":
            speed = 2.0 * p["u_in"] * (1.0 - 4.0 * (self.xy[0] ** 2 + self.xy[1] ** 2) / p["d_in"] ** 2)
        u = speed * self.normal
        if p["noise_amp"]:
            u = u + p["noise_amp"] * p["u_in"] * self._noise(p["noise_seed"])
        if self.t < p["inlet_ramp"]:
            s = self.t / p["inlet_ramp"]
            u = u * (s * s * (3.0 - 2.0 * s))
        return torch.where(inlet, rho_f, 1.0), torch.where(inlet, u, u_f)

    def _noise(self, seed):
        """Uniform variates in [-1, 1) of (seed, step, node, component) by SplitMix64 hashing."""
        def mix(v):
            z = v + np.uint64(0x9e3779b97f4a7c15)
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xbf58476d1ce4e5b9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94d049bb133111eb)
            return z ^ (z >> np.uint64(31))

        node = self.box[self.nodes].cpu().numpy().astype(np.uint64) << np.uint64(2)
        h = mix(np.array([seed], dtype=np.uint64))
        h = mix(np.array([self.t], dtype=np.uint64) + h)
        r = [(mix((node | np.uint64(a)) + h) >> np.uint64(40)).astype(np.float64) / 8388608.0 - 1.0 for a in range(3)]
        return torch.from_numpy(np.stack(r)).to(self.dev)

    def _interpolate(self, g):
        """Bouzidi's rule on the gathered values g of the cells with wall distances."""
        cells, wall, q = self.q
        h, own = g[:, cells], self.f[:, cells]
        new = h.clone()
        for i in range(27):
            near = 2.0 * q[i] * h[i] + (1.0 - 2.0 * q[i]) * h[26 - i]
            far = h[i] / (2.0 * q[i]) + (1.0 - 1.0 / (2.0 * q[i])) * own[i]
            v = torch.where(q[i] < 0.5, torch.where(wall[26 - i], h[i], near), far)
            new[i] = torch.where(wall[i] & (q[i] != 0.5), v, h[i])
        g[:, cells] = new

    def step(self, sample=None):
        """One time step; sample(slice, rho, u, sigma) sees each cell's moments and viscous stress."""
        self.t += 1
        flat, n = self.f.reshape(-1), self.n
        g = torch.empty_like(self.f)
        for i in range(27):
            torch.index_select(flat, 0, self.src[i], out=g[i])
        if self.q is not None:
            self._interpolate(g)
        rho, u, sec = [], [], []
        for b in range(0, n, self.CHUNK):
            e = slice(b, min(n, b + self.CHUNK))
            r, v = self.moments(g[:, e])
            g[:, e], s = self.collide(g[:, e], r, v)
            rho.append(r), u.append(v)
            if sample:
                sec.append(s)
        rho, u = torch.cat(rho), torch.cat(u, 1)
        sec = torch.cat(sec, 1) if sample else None
        if self.nodes.numel():
            k, j = self.nodes, self.partner
            rf, uf = rho[j], u[:, j]
            rb, ub = self._inlet(rf, uf)
            g[:, k] = self.equilibrium(rb, ub) + g[:, j] - self.equilibrium(rf, uf)
            rho[k], u[:, k] = rb, ub
            if sample:
                sec[:, k] = sec[:, j]
        self.f = g
        if sample:
            sample(rho, u, -(1.0 - 0.5 * self.omega) * sec)


def _plain_steps(case, steps):
    """About how long exact() takes, in seconds."""
    return steps * max(1.5e-3, 4.0e-9 * _cells(case))


def _exact_moments(lat):
    rho, u = lat.moments(lat.f)
    return [rho, u.T.contiguous()]


def exact(case, seed):
    if case["kind"] == "serving":
        out = []
        for flags, steps, precision, p in _requests(case, seed):
            lat = _Plain(flags, False, _omega(p["u_char"] * p["L_char"] / p["Re"]), params=p)
            lat.start(np.ones(lat.n), np.zeros((lat.n, 3)))
            for _ in range(steps):
                lat.step()
            out.append(_exact_moments(lat))
        return out
    if _plain_steps(case, case["steps"]) > 15.0:
        return None
    if case["kind"] == "vortex":
        n = case["n"]
        lat = _Plain(I.box_flags(n, n, n), True, _omega(_vortex_nu(case)), _ghost(case))
        lat.start(*_fields(case, lat.n, seed))
        for _ in range(case["steps"]):
            lat.step()
        return _exact_moments(lat)
    geometry = (case["kind"], case["D"], case["d"], case["length"])
    p = _params(case, seed)
    wall_q = _wall_q(*geometry) if case.get("walls") == "smooth" else None
    lat = _Plain(_flags(*geometry), False, _omega(p["u_char"] * p["L_char"] / p["Re"]), params=p, wall_q=wall_q)
    if case["kind"] == "restart":
        lat.f = torch.from_numpy(np.ascontiguousarray(_populations(case, lat.n, seed).T)).to(lat.dev)
        for _ in range(case["steps"]):
            lat.step()
        return lat.f.T.contiguous()
    lat.start(*_fields(case, lat.n, seed))
    sums = {}

    def sample(rho, u, sigma):
        uu = torch.stack([u[a] * u[b] for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))])
        for k, v in (("u", u), ("uu", uu), ("sigma", sigma), ("rho", rho)):
            sums[k] = sums[k] + v if k in sums else v.clone()

    for _ in range(case["steps"]):
        lat.step(sample if case["stats"] != "none" else None)
    out = _exact_moments(lat)
    mean = {k: v / case["steps"] for k, v in sums.items()}
    if case["stats"] == "axial":
        out += [mean["u"][2], mean["uu"][2]]
    elif case["stats"] == "full":
        out += [mean["u"].T.contiguous(), mean["uu"].T.contiguous(), mean["sigma"].T.contiguous(), mean["rho"]]
    return out
