"""Workloads for timing the library, each through the calls a user's program makes.

A case advances runs of the sparse-grid PIC scheme (``Run.step``) and reads the
state back on the device, serves a batch of independent runs (``Server``), or
sorts positions by cell (``sg_cell_sort``).  The sizes are those of the
benchmark workloads and of the serving mix (2D levels 5..10, 3D levels 5..7,
2^16 to 2^24 particles), with odd particle counts among them.

Positions live in a periodic box, where 1 - eps and 0 are neighbours, so a
pass returns each particle's minimum-image displacement since the start
instead of its wrapped position, next to the velocities, the regular-grid
density and the energies.
"""
import math
import random

import numpy as np
import torch

from paper_2008_09441_gb300.sgpic import Run, Server, sg_cell_sort

DEV = "cuda"
# A multiple of both default sort periods (4 in 2D, 6 in 3D): every pass does
# the same number of sorts.
STEPS = 12


def listed():
    return [
        # The paper's verification size in double precision: latency and launches.
        dict(name="landau2d_n6_fp64", kind="steps", problem="landau", dim=2, n=6, np=65536, precision="fp64",
             steps=STEPS, field=True),
        # Small members of a parameter scan, particle counts that fill no vector or block.
        dict(name="landau2d_n8_odd", kind="steps", problem="landau", dim=2, n=8, np=300007, precision="fp32",
             steps=STEPS, field=True),
        dict(name="twostream3d_n5_odd", kind="steps", problem="twostream", dim=3, n=5, np=100003, precision="fp32",
             steps=STEPS, field=False),
        # The headline benchmark: 2D Landau damping on the 1024^2 grid.
        dict(name="landau2d_n10", kind="steps", problem="landau", dim=2, n=10, np=4194304, precision="fp32",
             steps=STEPS, field=False),
        # 2D annulus in a magnetic field: Boris push, particles in a small part of the box.
        dict(name="diocotron2d_n9", kind="steps", problem="annulus", dim=2, n=9, np=8388608, precision="fp32",
             steps=STEPS, field=False),
        # 3D two-stream instability at full size: the largest run.
        dict(name="twostream3d_n7", kind="steps", problem="twostream", dim=3, n=7, np=16777216, precision="fp32",
             steps=STEPS, field=False),
        # 3D Penning trap: few particles per cell, external field, magnetic field.
        dict(name="penning3d_n7", kind="steps", problem="penning", dim=3, n=7, np=2097152, precision="fp32",
             steps=STEPS, field=False),
        # The paper's filter mode on its cell-centred grids: one solve on the regular grid.
        dict(name="landau2d_n10_filter_cell", kind="steps", problem="landau", dim=2, n=10, np=2000003,
             precision="fp32", mode="filter", centring="cell", steps=STEPS, field=False),
        # Adaptive truncation (Algorithm 1 before every field solve), as in the paper's two experiments.
        dict(name="diocotron_paper_n9_adaptive", kind="steps", problem="diocotron_paper", dim=2, n=9, np=1310720,
             precision="fp32", tau="adaptive", steps=4, field=False),
        dict(name="penning3d_n6_adaptive", kind="steps", problem="penning", dim=3, n=6, np=262144,
             precision="fp32", tau="adaptive", centring="cell", steps=4, field=False),
        # Serving: independent 2D and 3D runs submitted together, advanced tick by tick, results fetched.
        dict(name="serve_mix", kind="serve", mix=7, runs=8, max_log2=19, steps=20),
        # The stand-alone cell-key sort.
        dict(name="cell_sort_2d_n10", kind="sort", dim=2, n=10, np=4194304, precision="fp32"),
    ]


def _log_int(rng, lo_log2, hi_log2):
    return int(round(2.0 ** rng.uniform(lo_log2, hi_log2)))


def draw(rng):
    kind = rng.choices(["steps", "fp64", "adaptive", "serve", "sort"], weights=[10, 2, 2, 1, 2])[0]
    dim = rng.choice([2, 3])
    if kind == "sort":
        return dict(kind="sort", dim=dim, n=rng.randint(5, 10) if dim == 2 else rng.randint(4, 7),
                    np=_log_int(rng, 16, 23), precision=rng.choice(["fp32", "fp64"]))
    if kind == "serve":
        return dict(kind="serve", mix=rng.randint(1, 10 ** 6), runs=rng.randint(3, 8), max_log2=rng.choice([17, 18, 19]),
                    steps=20)
    problem = rng.choice(["landau", "annulus", "diocotron_paper"] if dim == 2 else ["twostream", "penning"])
    if kind == "fp64":
        return dict(kind="steps", problem=problem, dim=dim, n=rng.randint(5, 8) if dim == 2 else 5,
                    np=_log_int(rng, 14, 19), precision="fp64", steps=STEPS, field=dim == 2)
    if kind == "adaptive":
        return dict(kind="steps", problem="diocotron_paper" if dim == 2 else "penning", dim=dim,
                    n=rng.randint(7, 9) if dim == 2 else rng.randint(5, 6), np=_log_int(rng, 17, 20),
                    precision="fp32", tau="adaptive", steps=4, field=False)
    return dict(kind="steps", problem=problem, dim=dim, n=rng.randint(5, 10) if dim == 2 else rng.randint(5, 7),
                np=_log_int(rng, 16, 23), precision="fp32", steps=STEPS, field=False,
                tau=rng.choices([1, 2, 3], weights=[3, 1, 1])[0],
                mode=rng.choices(["combine", "filter"], weights=[4, 1])[0],
                centring=rng.choices(["node", "cell"], weights=[3, 1])[0])


# ---------------------------------------------------------------- inputs
def _box(case, k=None):
    """Box length, time step, B, external field and estimator settings of a problem."""
    p = case["problem"]
    if p == "landau":
        return dict(L=2.0 * math.pi / (k or 0.5), dt=0.05, B=(0.0, 0.0, 0.0), eext=(0.0, 0.0, 0.0))
    if p == "twostream":
        return dict(L=2.0 * math.pi / (k or 0.2), dt=0.05, B=(0.0, 0.0, 0.0), eext=(0.0, 0.0, 0.0))
    if p == "annulus":
        return dict(L=1.0, dt=0.05, B=(0.0, 0.0, 1.0), eext=(0.0, 0.0, 0.0))
    if p == "penning":
        L = 20.0
        return dict(L=L, dt=0.05, B=(0.0, 0.0, 5.0), eext=(-15.0 / L, -15.0 / L, 30.0 / L), alpha=0.005, pc_ref=1.0)
    return dict(L=22.0, dt=0.02, B=(0.0, 0.0, 5.0), eext=(0.0, 0.0, 0.0), alpha=0.01, pc_ref=5.0)


def _particles(case, seed, k=None, amplitude=None):
    """Positions (fractions of the box), velocities and charges, one row per axis, in the run's precision."""
    d, N, p = case["dim"], case["np"], case["problem"]
    L = _box(case, k)["L"]
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    rand = lambda *s: torch.rand(*s, generator=g, device=DEV, dtype=torch.float64)  # noqa: E731
    randn = lambda *s: torch.randn(*s, generator=g, device=DEV, dtype=torch.float64)  # noqa: E731
    v = randn(d, N)
    if p == "landau":
        u = rand(d, N)
        w = -(L ** d / N) * (1.0 + (0.05 if amplitude is None else amplitude) * torch.cos(2.0 * math.pi * u[0]))
    elif p == "twostream":
        u = rand(d, N)
        v *= 0.3
        v[0] += torch.where(rand(N) < 0.5, 3.0, -3.0)
        w = -(L ** d / N) * (1.0 + (1e-3 if amplitude is None else amplitude) * torch.cos(2.0 * math.pi * u[0]))
    elif p == "annulus":
        a, b = 0.3, 0.4
        r = torch.sqrt(a * a + (b * b - a * a) * rand(N))
        th = 2.0 * math.pi * rand(N)
        u = torch.stack([0.5 + r * torch.cos(th), 0.5 + r * torch.sin(th)])
        area = math.pi * (b * b - a * a)
        w = (-0.1 * area / N) * (1.0 + 0.01 * torch.cos(3.0 * th))
        # cold, drifting with E x B in the annulus' own radial field
        er = (-0.1 * (r * r - a * a) / 2.0 + 0.1 * area * r * r / 2.0) / r
        v = torch.stack([er * torch.sin(th), -er * torch.cos(th)])
    elif p == "penning":
        sd = torch.tensor([[0.15], [0.05], [0.2]], device=DEV, dtype=torch.float64)
        u = 0.5 + sd * randn(3, N)
        w = torch.full((N,), -1562.5 / N, device=DEV, dtype=torch.float64)
    else:  # the paper's hollow diocotron profile
        r = 0.25 + 0.03 * randn(N)
        th = 2.0 * math.pi * rand(N)
        u = torch.stack([0.5 + r * torch.cos(th), 0.5 + r * torch.sin(th)])
        w = torch.full((N,), -400.0 / N, device=DEV, dtype=torch.float64)
    u = u - torch.floor(u)
    dt = torch.float32 if case["precision"] == "fp32" else torch.float64
    u, v, w = u.to(dt), v.to(dt).contiguous(), w.to(dt)
    return torch.where(u >= 1, torch.zeros_like(u), u).contiguous(), v, w


def _mix(case):
    """The serving mix: each run's sizes and parameters."""
    rng = random.Random(case["mix"])
    runs = []
    for _ in range(case["runs"]):
        dim = rng.choice([2, 3])
        runs.append(dict(dim=dim, n=rng.randint(5, 10) if dim == 2 else rng.randint(5, 7),
                         np=_log_int(rng, 16, case["max_log2"]), problem="landau" if dim == 2 else "twostream",
                         precision="fp32", k=rng.uniform(0.3, 0.6), amplitude=10.0 ** rng.uniform(-3, -1)))
    return runs


def prepare(case, seed):
    if case["kind"] == "sort":
        u, _, _ = _particles(dict(case, problem="landau"), seed)
        return dict(case=case, u=u)
    if case["kind"] == "serve":
        runs = []
        for i, r in enumerate(_mix(case)):
            u, v, w = (x.cpu().numpy() for x in _particles(r, seed * 64 + i, r["k"], r["amplitude"]))
            runs.append(dict(r, L=_box(r, r["k"])["L"], u=u, v=v, w=w))
        return dict(case=case, runs=runs)
    u, v, w = _particles(case, seed)
    b = _box(case)
    d = case["dim"]
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    tau = case.get("tau", 1)
    run = Run((b["L"],) * d, case["n"], list(u), list(v), w, b["dt"], tau=-1 if tau == "adaptive" else tau,
              precision=case["precision"], B=b["B"], eext_lin=b["eext"], alpha=b.get("alpha", 0.01),
              pc_ref=b.get("pc_ref", 5.0), mode=case.get("mode", "combine"), centring=case.get("centring", "node"),
              stream=stream.cuda_stream)
    return dict(case=case, run=run, stream=stream, u0=u, u=torch.empty_like(u), v=torch.empty_like(v),
                w=torch.empty_like(w), rho=torch.empty((1 << case["n"],) * d, dtype=u.dtype, device=DEV))


# ---------------------------------------------------------------- one pass
def run(state):
    case = state["case"]
    if case["kind"] == "sort":
        keys, perm, counts = sg_cell_sort(list(state["u"]), case["n"], 0 if case["precision"] == "fp32" else 1)
        return dict(keys=keys, perm=perm, counts=counts)
    if case["kind"] == "serve":
        server = Server(16 << 30, 64)
        tickets = [server.submit((r["L"],) * r["dim"], r["n"], list(r["u"]), list(r["v"]), r["w"], 0.05, case["steps"])
                   for r in state["runs"]]
        while server.tick():
            pass
        out = []
        for t, r in zip(tickets, state["runs"]):
            _, diag = server.poll(t)
            u, v, _ = server.result(t)
            d = u.T - r["u"]
            d -= np.rint(d)
            out.append((d, v.T, _energies(diag, np.float32)))
        server.close()
        return out
    r, u = state["run"], state["u"]
    with torch.cuda.stream(state["stream"]):
        r.step(case["steps"])
        r.particles_device(list(u), list(state["v"]), state["w"])
        r.density_copy(state["rho"], to_run=False)
        moved = u - state["u0"]
        moved -= moved.round()
        real = np.float32 if case["precision"] == "fp32" else np.float64
        out = dict(moved=moved, v=state["v"], rho=state["rho"], energies=_energies(r.diagnostics(), real))
        if case["field"]:
            out["field"] = r.field().astype(real)
    return out


def _energies(diag, real):
    return np.array([diag["field_energy"], diag["kinetic_energy"], diag["charge_combined"]], dtype=real)


# ---------------------------------------------------------------- bytes and operations
def work(case):
    if case["kind"] == "sort":
        rs = 4 if case["precision"] == "fp32" else 8
        return dict(bytes=case["np"] * (case["dim"] * rs + 8) + 4 * 2 ** (case["dim"] * case["n"]),
                    flops=case["np"] * 8.0)
    if case["kind"] == "serve":
        total = dict(bytes=0.0, flops=0.0)
        for r in _mix(case):
            w = work(dict(r, kind="steps", steps=case["steps"]))
            total = {k: total[k] + w[k] for k in total}
        return total
    d, N, rs = case["dim"], case["np"], 4 if case["precision"] == "fp32" else 8
    nodes = 2 ** (d * case["n"])
    # every step: each particle's position, velocity and charge read, position
    # and velocity written; the regular density and field written and read.
    # The read-back writes the final state once.
    step = N * (4 * d + 1) * rs + 2 * nodes * (1 + d) * rs
    out = N * (2 * d + 1) * rs + nodes * rs
    corner = 2 ** d
    flops = N * (corner * (2 * d + 2 * d + 2) + 12 * d) + nodes * 8 * d
    if case.get("mode") == "filter" or case.get("tau") == "adaptive":
        flops += nodes * 5 * d * case["n"] * (2 + d)
    return dict(bytes=float(case["steps"] * step + out), flops=float(case["steps"] * flops))


# ---------------------------------------------------------------- the same in 64 bits
def _grids(d, n, tau):
    """(levels, coefficient) of the truncated combination technique."""
    out = []
    for q in range(d):
        c = (-1) ** q * math.comb(d - 1, q)
        for i in range(tau, n + 1):
            for j in range(tau, n + 1):
                if d == 2 and i + j == n + tau - q:
                    out.append(((i, j), c))
                elif d == 3 and tau <= n + 2 * tau - q - i - j <= n:
                    out.append(((i, j, n + 2 * tau - q - i - j), c))
    return out


class _Exact:
    """The scheme in float64: arrays are indexed [i_d, .., i_1] (x fastest)."""

    def __init__(self, case, b):
        self.d, self.n, self.N = case["dim"], case["n"], 1 << case["n"]
        self.L, self.b, self.case = b["L"], b, case
        self.cell = case.get("centring", "node") == "cell"
        self.P = {}

    def prolong(self, l):
        """(N, 2^l) linear interpolation from level-l to level-n nodes."""
        if l not in self.P:
            off = 0.5 if self.cell else 0.0
            x = ((torch.arange(self.N, device=DEV, dtype=torch.float64) + off) / self.N)[:, None]
            y = ((torch.arange(1 << l, device=DEV, dtype=torch.float64) + off) / (1 << l))[None]
            dist = (x - y).abs()
            dist = torch.minimum(dist, 1.0 - dist)
            m = torch.clamp(1.0 - dist * (1 << l), min=0.0)
            if l == 0:
                m = torch.ones_like(m)
            self.P[l] = m
        return self.P[l]

    def along(self, a, mats):
        """Apply mats[m] (out, in) along axis x_m of a."""
        for m, mat in enumerate(mats):
            dim = a.dim() - 1 - m
            a = torch.movedim(torch.tensordot(mat, a, dims=([1], [dim])), 0, dim)
        return a

    def restrict(self, rho, l):
        return self.along(rho, [self.prolong(k).T * (2.0 ** k / self.N) for k in l])

    def corners(self, u):
        s = u * self.N - (0.5 if self.cell else 0.0)
        c = torch.floor(s)
        f = s - c
        c = c.to(torch.int64)
        for corner in range(1 << self.d):
            w, idx, stride = 1.0, 0, 1
            for m in range(self.d):
                bit = (corner >> m) & 1
                w = w * (f[m] if bit else 1.0 - f[m])
                idx = idx + ((c[m] + bit) % self.N) * stride
                stride *= self.N
            yield idx, w

    def deposit(self, u, q):
        rho = torch.zeros(self.N ** self.d, device=DEV, dtype=torch.float64)
        for idx, w in self.corners(u):
            rho.index_add_(0, idx, q * w)
        return (rho * (self.N / self.L) ** self.d).reshape((self.N,) * self.d)

    def waves(self, shape):
        """k_m along axis x_m, broadcastable, and the Nyquist mask of each axis."""
        ks, nyq = [], []
        for m in range(self.d):
            size = shape[self.d - 1 - m]
            i = torch.arange(size, device=DEV)
            k = 2.0 * math.pi / self.L * torch.where(i < size // 2, i, i - size).to(torch.float64)
            view = [1] * self.d
            view[self.d - 1 - m] = size
            ks.append(k.view(view))
            nyq.append((i == size // 2).view(view))
        return ks, nyq

    def poisson(self, rho):
        ks, nyq = self.waves(rho.shape)
        k2 = sum(k * k for k in ks)
        phi = torch.where(k2 > 0, torch.fft.fftn(rho) / torch.where(k2 > 0, k2, torch.ones_like(k2)), 0.0)
        return [torch.fft.ifftn(torch.where(z, torch.zeros_like(phi), -1j * k * phi)).real for k, z in zip(ks, nyq)]

    def field(self, rho, tau):
        if self.case.get("mode", "combine") == "filter":
            f = sum(c * self.along(self.restrict(rho, l), [self.prolong(k) for k in l])
                    for l, c in _grids(self.d, self.n, tau))
            return torch.stack(self.poisson(f))
        E = torch.zeros((self.d,) + rho.shape, device=DEV, dtype=torch.float64)
        for l, c in _grids(self.d, self.n, tau):
            mats = [self.prolong(k) for k in l]
            for m, e in enumerate(self.poisson(self.restrict(rho, l))):
                E[m] += c * self.along(e, mats)
        return E

    def estimate(self, rho, npart, q_total):
        """The truncation parameter of the paper's Algorithm 1 (printed constants)."""
        d, n, N, L = self.d, self.n, self.N, self.L
        z = torch.fft.fftn(rho) / N ** d
        frac = self.b["alpha"] * math.sqrt(self.b["pc_ref"] / (npart / N ** d))
        z = torch.where(z.abs() >= frac * z.abs().max(), z, torch.zeros_like(z))
        ks, _ = self.waves(rho.shape)

        def top(axes):
            f = z
            for m in axes:
                f = f * ks[m] ** 2
            return float((torch.fft.ifftn(f) * N ** d).real.abs().max())

        kappa = [0.25 * top([m]) for m in range(d)]
        pairs = [[0, 1]] if d == 2 else [[0, 1], [1, 2], [2, 0]]
        beta = sum(top(p) / 72.0 for p in pairs)
        gamma = top([0, 1, 2]) / 864.0 if d == 3 else 0.0
        sigma = math.sqrt((2.0 / 3.0) ** d * abs(q_total) * float(rho.abs().max()))
        h, best = L / N, None
        for t in range(1, (n - 3 if d == 2 else n - 2) + 1):
            m = n - t
            if d == 2:
                g = h * h * (sum(kappa) + beta * L * L * 2.0 ** (-2 * t) * (5 * m + 1))
                s = sigma * 2.0 ** (0.5 * (t - 1)) * (m * (1 + math.sqrt(2)) + math.sqrt(2)) / math.sqrt(npart * h * L)
            else:
                g = h * h * (sum(kappa) + beta * L * L * 2.0 ** (-2 * t) * (5 * m + 1)
                             + gamma * L ** 4 * 2.0 ** -(4 * t + 1) * (25 * m * m - 5 * m + 2))
                s = sigma * 2.0 ** (t - 2) * ((3 + math.sqrt(2)) * m * m + (5 + math.sqrt(2)) * m + 4) \
                    / math.sqrt(npart * h * L * L)
            if best is None or g + s < best[0]:
                best = (g + s, t)
        return best[1]

    def kick(self, u, v, E, dt):
        """Half kick, Boris rotation, half kick (q/m = -1)."""
        F = torch.zeros_like(u)
        for idx, w in self.corners(u):
            for m in range(self.d):
                F[m] += w * E[m].reshape(-1)[idx]
        for m in range(self.d):
            if self.b["eext"][m]:
                F[m] += self.b["eext"][m] * self.L * (u[m] - 0.5)
        F *= -0.5 * dt
        v = v + F
        t = -0.5 * dt * self.b["B"][2]  # the field is along z
        if t:
            s = 2.0 * t / (1.0 + t * t)
            px, py = v[0] + v[1] * t, v[1] - v[0] * t
            v[0], v[1] = v[0] + py * s, v[1] - px * s
        return v + F

    def advance(self, u, v, q, steps):
        tau, total = self.case.get("tau", 1), float(q.sum())

        def solve():
            rho = self.deposit(u, q)
            t = self.estimate(rho, u.shape[1], total) if tau == "adaptive" else tau
            return rho, self.field(rho, t)

        dt = self.b["dt"]
        moved = torch.zeros_like(u)
        rho, E = solve()
        v = self.kick(u, v, E, -0.5 * dt)
        ke = 0.0
        for _ in range(steps):
            old = v
            v = self.kick(u, v, E, dt)
            ke = float(-0.5 * (q * (old * v).sum(0)).sum())
            moved += v * (dt / self.L)
            u = u + v * (dt / self.L)
            u = u - torch.floor(u)
            rho, E = solve()
        moved -= moved.round()
        fe = 0.5 * (self.L / self.N) ** self.d * float((E * E).sum())
        return moved, v, rho, E, np.array([fe, ke, total])


def exact(case, seed):
    if case["kind"] == "sort":
        return None  # whole numbers
    if case["kind"] == "serve":
        out = []
        for i, r in enumerate(_mix(case)):
            u, v, w = (x.double() for x in _particles(r, seed * 64 + i, r["k"], r["amplitude"]))
            moved, v, _, _, en = _Exact(r, _box(r, r["k"])).advance(u, v, w, case["steps"])
            out.append((moved, v, en))
        return out
    u, v, w = (x.double() for x in _particles(case, seed))
    moved, v, rho, E, en = _Exact(case, _box(case)).advance(u, v, w, case["steps"])
    out = dict(moved=moved, v=v, rho=rho, energies=en)
    if case["field"]:  # indexed [m, i_1, .., i_d]
        out["field"] = E.permute((0,) + tuple(range(case["dim"], 0, -1))).contiguous()
    return out
