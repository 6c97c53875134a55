"""Performance cases of the N-phase solver: what a user has it do, and how much work that is.

A pass advances a simulation by a number of time steps and reads its macroscopic fields
(``Solver.step`` and ``Solver.moments``), which is the loop of every run of this package: some
steps, then the fields for a plot or a measurement. The whole-run case also starts the simulation
from volume fractions and reads the conservation diagnostics; the ensemble advances many grids
with ``Batch``. Grids, phase numbers, densities, walls, gradient schemes and storage forms are
those of the workloads, tests and benchmark of this repository; ``draw`` spreads them over the
ranges in between, odd sizes among them.

Fields come back as the solver computes them: FP64 for the FP64 form, FP32 for the forms whose
arithmetic is FP32 (the API hands every field out in FP64; narrowing those loses nothing).

``exact`` is the same model in FP64, written with torch operations on whole fields.
"""
import math

import numpy as np
import torch

from paper_1904_12553_gb300 import Batch, Solver, workloads
from paper_1904_12553_gb300 import binding

DEV = "cuda"


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------

def _grid(name, N, nx, ny, precision, steps, *, nz=0, wall=0, rho="", scheme=0, gravity=0.0,
          layers=1, drops=4, speed=0.01, start=False):
    """One grid. rho: "" for equal pure-phase densities, else "10,1,5"; nz = 0: two dimensions;
    layers: phases stacked in y (the others are drops); start: the pass begins at the volume
    fractions."""
    return {"name": name, "kind": "grid", "N": N, "nx": nx, "ny": ny, "nz": nz,
            "precision": precision, "steps": steps, "wall": wall, "rho": rho, "scheme": scheme,
            "gravity": gravity, "layers": layers, "drops": drops, "speed": speed, "start": start}


def listed():
    return [
        # A whole small run: the three-phase static drops of the first benchmark set, started,
        # stepped, with its conservation diagnostics and fields. One step is a few microseconds:
        # launches and latency count.
        _grid("drops_128_fp64", 3, 128, 128, "fp64", 400, layers=1, drops=2, speed=0.001,
              start=True),
        # The paper's liquid lens: 150 nodes wide (no whole tiles, rows not 16-byte multiples in
        # FP32), density ratio 10:1:5, walls.
        _grid("lens_150_fp64", 3, 150, 150, "fp64", 200, wall=1, rho="10,1,5", layers=2, drops=1,
              speed=0.002),
        # The paper's five-phase run: droplets and a bubble under gravity, mixed gradient scheme.
        _grid("five_phase_200x320_fp64", 5, 200, 320, "fp64", 100, wall=1, rho="6,4,1,2,3",
              scheme=1, gravity=1e-5, layers=2, drops=3, speed=0.002),
        # The paper's puddle: lens under gravity with unequal densities, FP32.
        _grid("puddle_400x200_fp32", 3, 400, 200, "fp32", 200, wall=1, rho="3,1,6",
              gravity=5e-5, layers=2, drops=1, speed=0.002),
        # The benchmark set's lens between walls, FP32.
        _grid("lens_256_fp32", 3, 256, 256, "fp32", 400, wall=1, layers=2, drops=1),
        # Colliding drops, four phases, 16-bit storage of the moving populations.
        _grid("collision_512_bf16", 4, 512, 512, "bf16", 200, layers=1, drops=3),
        # The headline: five phases, droplets and interfaces, FP32.
        _grid("droplets_2048_fp32", 5, 2048, 2048, "fp32", 40, layers=3, drops=8),
        # The same system in FP64, as it is run for reference solutions.
        _grid("droplets_1024_fp64", 5, 1024, 1024, "fp64", 20, layers=3, drops=8),
        # A domain whose sides are set by the physics and not by a tile: odd in x and y.
        _grid("layers_1501x997_fp32", 4, 1501, 997, "fp32", 40, layers=2, drops=4),
        # A parameter sweep: independent small grids of several sizes and phase numbers.
        {"name": "ensemble_48_fp32", "kind": "batch", "cases": 48, "smin": 64, "smax": 512,
         "grain": 64, "steps": 60, "pipelined": True},
        # Three dimensions: the benchmark's box of spheres, FP32.
        _grid("spheres_256_fp32", 3, 256, 256, "fp32", 10, nz=256, layers=1, drops=2),
        # A smaller box with walls and 16-bit storage.
        _grid("spheres_128_bf16", 3, 128, 128, "bf16", 20, nz=128, wall=1, layers=1, drops=2),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: sizes log-uniform, half of them as they fall (odd ones too),
    half rounded to whole tiles; a cost of at most the largest listed case's."""
    kind = rng.random()
    if kind < 0.12:
        grain = rng.choice([8, 16, 32, 64])
        return {"kind": "batch", "cases": rng.randint(8, 48), "smin": 48 + 8 * rng.randint(0, 4),
                "smax": 8 * rng.randint(24, 64), "grain": grain, "steps": rng.randint(10, 60),
                "pipelined": rng.random() < 0.75}
    whole = rng.random() < 0.5
    side = (lambda v: max(32, (v + 16) // 32 * 32)) if whole else (lambda v: v)
    N = rng.randint(2, 5)
    unequal = rng.random() < 0.35
    wall = int(rng.random() < 0.5)
    if kind < 0.27:
        precision = rng.choice(["fp64", "fp32", "fp32", "bf16", "fp16"])
        top = 80 if precision == "fp64" or unequal else 200
        N = min(N, 4)
        nx, ny, nz = (side(_log(rng, 24, top)) for _ in range(3))
        scheme = 0
        cost = nx * ny * nz * (8 if unequal else 1)
    else:
        precision = rng.choice(["fp64", "fp64", "fp32", "fp32", "fp32", "bf16", "fp16"])
        top = 700 if precision == "fp64" else 2048
        nx, ny, nz = side(_log(rng, 48, top)), side(_log(rng, 48, top)), 0
        scheme = int(rng.random() < 0.15)
        cost = nx * ny * (2 if unequal or scheme else 1)
    cost *= (12 if precision == "fp64" else 1) * N / 5.0
    steps = max(8, min(400, int(10 ** rng.uniform(7.2, 8.1) / cost)))
    rho = ",".join(str(rng.randint(1, 6)) for _ in range(N - 1)) + ",7" if unequal else ""
    layers = 1 if N == 2 else rng.randint(1, 2)
    c = _grid("", N, nx, ny, precision, steps, nz=nz, wall=wall, rho=rho, scheme=scheme,
              gravity=1e-5 if unequal and wall else 0.0, layers=layers, drops=N - layers,
              speed=0.002 if unequal else 0.01, start=rng.random() < 0.2)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _params(case, rng):
    N, nx, ny, nz = case["N"], case["nx"], case["ny"], case["nz"]
    if case["rho"]:
        rho, sigma = [float(r) for r in case["rho"].split(",")], 0.01
    else:
        rho, sigma = None, np.zeros((N, N))
        for k in range(N):
            for l in range(k + 1, N):
                sigma[k, l] = sigma[l, k] = rng.uniform(0.95e-3, 1.05e-3)
    kw = dict(rho=rho, tau=[float(rng.uniform(0.7, 0.85)) for _ in range(N - 1)],
              tau_g=float(rng.uniform(0.7, 0.85)), mobility=0.1, wall_y=case["wall"],
              precision=case["precision"], grad_scheme=case["scheme"])
    g = -case["gravity"]
    if nz:
        return workloads.base_params3(N, nx, ny, nz, sigma, gravity=(0.0, g, 0.0), **kw)
    return workloads.base_params(N, nx, ny, sigma, gravity=(0.0, g), **kw)


def _step(d):
    return 0.5 + 0.5 * torch.tanh(d * 0.5)  # tanh(d / (sqrt(2) eta)), eta = sqrt(2)


def _start(case, rng):
    """Volume fractions c0[N][(nz)][ny][nx] (layers in y, seeded drops) and a smooth velocity."""
    N, wall, L = case["N"], case["wall"], case["layers"]
    size = ([case["nz"]] if case["nz"] else []) + [case["ny"], case["nx"]]
    D = len(size)
    axes = []  # coordinates, x first
    for d in range(D):
        shape = [1] * D
        shape[D - 1 - d] = -1
        axes.append(torch.arange(size[D - 1 - d], dtype=torch.float64, device=DEV).view(shape))
    c = torch.zeros([N] + size, dtype=torch.float64, device=DEV)
    # drops, one to a cell of a regular division of the box along its longest axis
    nd = case["drops"] if N > L else 0
    long = max(range(D), key=lambda d: size[D - 1 - d])
    for j in range(nd):
        r2 = 0.0
        cell = size[D - 1 - long] / nd
        R = min([cell] + size) * rng.uniform(0.22, 0.3)
        for d in range(D):
            n = size[D - 1 - d]
            at = (j + rng.uniform(0.45, 0.55)) * cell if d == long else n * rng.uniform(0.42, 0.58)
            dist = axes[d] - at
            if not (wall and d == 1):
                dist = dist - n * torch.round(dist / n)
            r2 = r2 + dist * dist
        c[L + j % (N - L)] += _step(R - torch.sqrt(r2))
    free = 1.0 - c.sum(0)
    rest = torch.ones(size, dtype=torch.float64, device=DEV)
    y, ny = axes[1], case["ny"]
    for l in range(1, L):
        band = 0.0
        for m in (0,) if wall else (-1, 0, 1):
            band = band + _step(y + m * ny - ny * l / L) - (
                0.0 if wall and l == L - 1 else _step(y + m * ny - ny * (l + 1) / L + (0.5 if l == L - 1 else 0.0)))
        rest = rest - band
        c[l] = band * free
    c[0] = rest * free
    u = torch.empty([D] + size, dtype=torch.float64, device=DEV)
    for d in range(D):
        e = (d + 1) % D
        u[d] = case["speed"] * torch.sin(
            axes[e] * (2 * math.pi / size[D - 1 - e]) + rng.uniform(0, 2 * math.pi))
    return c, u


def _batch_grids(case, rng):
    sides = list(range(case["smin"], case["smax"] + 1, case["grain"]))
    grids = []
    for i in range(case["cases"]):
        # the first ones take the sizes in turn, so that every seed has about the same work
        side = sides[i % len(sides)]
        N = 3 + i % 3
        grids.append(_grid("", N, side, side, "fp32", case["steps"], wall=i % 2,
                           layers=1 + i % 2, drops=N - 1 - i % 2, speed=0.005))
    return [(g, _params(g, rng)) + _start(g, rng) for g in grids]


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    if case["kind"] == "batch":
        grids = _batch_grids(case, rng)
        b = Batch([p for _, p, _, _ in grids])
        # the schedules that autotune() finds best on ensembles with and without tensor maps
        if case["pipelined"]:
            b.set_schedule(8, 2, pipelined=True, chunk=4)
        else:
            b.set_schedule(8, 2)
        for i, (_, _, c, u) in enumerate(grids):
            binding.lbm_nphase_batch_init(b.handle, i, c.data_ptr(), u.data_ptr(), 0.0)
        return {"case": case, "batch": b, "shapes": [(g["N"], g["ny"], g["nx"]) for g, _, _, _ in grids]}
    p = _params(case, rng)
    c, u = _start(case, rng)
    s = Solver(p)
    if case["start"]:
        return {"case": case, "solver": s, "c": c, "u": u}
    s.init(c, u)
    return {"case": case, "solver": s}


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        b = state["batch"]
        b.step(case["steps"])
        out = []
        for i, (N, ny, nx) in enumerate(state["shapes"]):
            f = torch.empty((N + 2, ny, nx), dtype=torch.float64, device=DEV)
            binding.lbm_nphase_batch_moments(b.handle, i, phi=f[0].data_ptr(),
                                             u=f[N - 1].data_ptr(), p=f[N + 1].data_ptr())
            out.append(f.float())
        return out
    s = state["solver"]
    fine = case["precision"] == "fp64"
    out = {}
    if case["start"]:
        s.init(state["c"], state["u"])
    s.step(case["steps"])
    if case["start"]:
        mass, ke, umax = s.diagnostics()
        out["mass"] = mass if fine else mass.astype(np.float32)
        out["ke"], out["umax"] = ke, umax
    for k, v in s.moments(numpy=False).items():
        out[k] = v if fine else v.float()
    return out


def _node_work(case):
    """Bytes of the state and operations of one node, as the paper's step needs them."""
    N, n = case["N"], case["N"] - 1
    three = case["nz"] > 0
    Q, D = (14, 3) if three else (8, 2)
    wide = 8 if case["precision"] == "fp64" else 4
    moving = {"fp64": 8, "fp32": 4, "bf16": 2, "fp16": 2}[case["precision"]]
    state = (n * Q + Q) * moving + (2 * n + D + (moving == 2)) * wide
    flops = (200 + n * (150 + 2 * n)) if three else (120 + n * (95 + 2 * n))
    if case["rho"]:
        flops += 60 + 30 * n
    fields = (2 * N + D + 1) * 8
    return state, flops, fields


def work(case):
    if case["kind"] == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        sides = list(range(case["smin"], case["smax"] + 1, case["grain"]))
        for i in range(case["cases"]):
            N, side = 3 + i % 3, sides[i % len(sides)]
            g = _grid("", N, side, side, "fp32", case["steps"])
            s, f, _ = _node_work(g)
            total["bytes"] += side * side * (2 * s + (N + 2) * 8)
            total["flops"] += side * side * f * case["steps"]
        return total
    V = case["nx"] * case["ny"] * max(1, case["nz"])
    s, f, m = _node_work(case)
    begin = (case["N"] + (3 if case["nz"] else 2)) * 8
    return {"bytes": float(V * (m + (begin if case["start"] else 2 * s))),
            "flops": float(V * f * case["steps"])}


# ---------------------------------------------------------------------------
# The model in 64 bits
# ---------------------------------------------------------------------------

class _Model:
    """The time step of the paper on whole fields (torch, FP64), D2Q9 or D3Q15. Fields are
    [(z)][y][x]; velocities are (x, y[, z])."""

    def __init__(self, p):
        self.p = p
        self.three = int(p.get("lattice", 0)) == 1
        if self.three:
            faces = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (-1, 0, 0), (0, -1, 0), (0, 0, -1)]
            corners = [(a, b, c) for a in (1, -1) for b in (1, -1) for c in (1, -1)]
            self.c = [(0, 0, 0)] + faces + corners
            self.w = [2 / 9] + [1 / 9] * 6 + [1 / 72] * 8
        else:
            self.c = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
            self.w = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
        self.D = 3 if self.three else 2
        self.opp = [self.c.index(tuple(-v for v in c)) for c in self.c]
        self.wall = bool(p["wall_y"])
        self.N = N = p["N"]
        n = self.n = N - 1
        rho = self.rho = np.array(p["rho"])
        self.gam = 1.0 / rho
        self.Gam = self.gam.sum()
        sig, eta = np.array(p["sigma"]), p["eta"]
        smin = min(sig[k, l] for k in range(N) for l in range(k + 1, N))
        beta2 = p["beta"] ** 2 if p["beta"] > 0 else 3 * math.sqrt(2) * smin * eta
        self.bulk = beta2 / eta ** 2
        pairs = [(i, j) for i in range(n) for j in range(i, n)]

        def L(i, k, l):  # Eqs. N15, N16
            if l == n:
                return 1.0 if i == k else rho[n] / (rho[i] + rho[n])
            if i == k:
                return rho[k] / (rho[k] + rho[n])
            return -rho[l] / (rho[l] + rho[n]) if i == l else 0.0

        A, b = [], []
        for k in range(N):
            for l in range(k + 1, N):
                A.append([L(i, k, l) * L(j, k, l) * (1 if i == j else 2) for i, j in pairs])
                b.append(4.5 * eta * eta / beta2 * sig[k, l] ** 2)
        x = np.linalg.solve(np.array(A), np.array(b))
        self.lam = np.zeros((n, n))
        for (i, j), v in zip(pairs, x):
            self.lam[i, j] = self.lam[j, i] = v
        tau = np.array(p["tau"])
        self.a = np.array(p["mobility"]) * 3.0 / (tau - 0.5)
        mul = 0.5 * (rho[:n] + rho[n])
        self.mul, self.off = mul, 0.5 * (rho[:n] - rho[n])
        self.K = 1.0 - N * self.gam[:n] / self.Gam
        self.kap = self.K * mul
        self.unequal = bool((rho != rho[0]).any())
        g = list(p["gravity"]) + [0.0]
        self.grav = g[:self.D]

    def at(self, f, c, times=1):
        """f at x + times c: periodic, the rows beyond a wall repeat the last one."""
        dims, shifts = [], []
        for d, v in enumerate(c):
            if v and not (d == 1 and self.wall):
                dims.append(-1 - d)
                shifts.append(-times * v)
        f = torch.roll(f, shifts, dims) if dims else f
        if self.wall and c[1]:
            ny = f.shape[-2]
            rows = torch.clamp(torch.arange(ny, device=f.device) + times * c[1], 0, ny - 1)
            f = f.index_select(f.dim() - 2, rows)
        return f

    def grad(self, f):
        """First derivatives along x, y[, z]: Eq. N31a or (scheme 1) Eq. N40."""
        out = [0.0] * self.D
        for k in range(1, len(self.c)):
            c = self.c[k]
            if self.p["grad_scheme"] == 1:
                back = tuple(-v for v in c)
                d = (-self.at(f, c, 2) + 5.0 * self.at(f, c) - 3.0 * f - self.at(f, back)) * 0.75
            else:
                d = self.at(f, c) * 3.0
            for e in range(self.D):
                if c[e]:
                    out[e] = out[e] + self.w[k] * c[e] * d
        return torch.stack(out)

    def lap(self, f):
        s = 0.0
        for k in range(1, len(self.c)):
            s = s + self.w[k] * self.at(f, self.c[k])
        return 6.0 * (s - (1.0 - self.w[0]) * f)

    def potentials(self, ph):
        n, N = self.n, self.N
        vp = [self.off[j] + self.mul[j] * ph[j] for j in range(n)]
        s = sum(self.gam[j] * vp[j] for j in range(n))
        c = [self.gam[k] / self.Gam * (1.0 - s) + (self.gam[k] * vp[k] if k < n else 0.0) for k in range(N)]
        rho = N / self.Gam + sum(self.K[i] * vp[i] for i in range(n))
        f = [x * (1.0 - x) * (1.0 - 2.0 * x) for x in c]
        fs = sum(self.gam[k] * f[k] for k in range(N))
        lp = [self.lap(ph[j]) for j in range(n)]
        C = []
        for i in range(n):
            hf = self.mul[i] * (self.gam[i] * f[i] - self.gam[i] / self.Gam * fs)
            C.append(self.bulk * hf - sum(self.lam[i, j] * lp[j] for j in range(n)))
        return torch.stack(c), rho, torch.stack(C)

    def start(self, c0, u0):
        n, N = self.n, self.N
        ph = torch.stack([(2.0 * (self.rho[i] * c0[i] - self.rho[n] * c0[n]) - (self.rho[i] - self.rho[n]))
                          / (self.rho[i] + self.rho[n]) for i in range(n)])
        _, rho, C = self.potentials(ph)
        Q = len(self.c)
        uu = sum(u0[d] * u0[d] for d in range(self.D))
        self.g = torch.zeros((Q,) + tuple(rho.shape), dtype=torch.float64, device=rho.device)
        self.h = torch.zeros((n, Q) + tuple(rho.shape), dtype=torch.float64, device=rho.device)
        for k in range(Q):
            cu = sum(self.c[k][d] * u0[d] for d in range(self.D))
            if k:
                self.g[k] = self.w[k] * rho * (3 * cu + 4.5 * cu * cu - 1.5 * uu)
            for i in range(n):
                self.h[i, k] = self.heq(k, i, ph[i], C[i], cu)
        self.pp, self.up = ph, u0.clone()

    def heq(self, k, i, ph, C, cu):
        if k == 0:
            return ph + (self.w[0] - 1.0) * self.a[i] * C
        return self.w[k] * (self.a[i] * C + 3.0 * ph * cu)

    def fields(self):
        n, D = self.n, self.D
        ph = self.h.sum(1)
        c, rho, C = self.potentials(ph)
        gp = torch.stack([self.grad(ph[i]) for i in range(n)])
        zero = torch.zeros((D,) + tuple(rho.shape), dtype=torch.float64, device=rho.device)
        gr, J = zero, zero
        if self.unequal:
            gr = sum(self.kap[i] * gp[i] for i in range(n))
            J = -sum(self.kap[i] * self.p["mobility"][i] * self.grad(C[i]) for i in range(n))
        F = torch.stack([rho * self.grav[d] + sum(C[i] * gp[i, d] for i in range(n)) for d in range(D)])
        m = torch.stack([sum(self.c[k][d] * self.g[k] for k in range(1, len(self.c)) if self.c[k][d])
                         for d in range(D)])
        u = (m + 0.5 * F) / rho
        uu = (u * u).sum(0)
        pr = (1 / 3) / (1 - self.w[0]) * (self.g[1:].sum(0) + 0.5 * (u * gr).sum(0)
                                          - self.w[0] * 1.5 * rho * uu)
        return ph, c, rho, C, gr, J, F, u, uu, pr

    def step(self):
        D, n = self.D, self.n
        ph, _, rho, C, gr, J, F, u, uu, pr = self.fields()
        tg = self.p["tau_g"]
        T = [[u[a] * F[b] + F[a] * u[b] + (u[a] * gr[b] + gr[a] * u[b]) / 3 + J[a] * u[b] / (tg - 0.5)
              for b in range(D)] for a in range(D)]
        trace = sum(T[a][a] for a in range(D)) / 3
        ugr = (u * gr).sum(0)
        jump = [[ph[i] * u[d] - self.pp[i] * self.up[d] for d in range(D)] for i in range(n)]
        for k, c in enumerate(self.c):
            cu = sum(c[d] * u[d] for d in range(D))
            if k:  # g_0 enters no output
                cF = sum(c[d] * F[d] for d in range(D))
                QT = sum(c[a] * c[b] * T[a][b] for a in range(D) for b in range(D)) - trace
                G = self.w[k] * (ugr + 3 * cF + 4.5 * QT)
                geq = self.w[k] * (3 * pr + rho * (3 * cu + 4.5 * cu * cu - 1.5 * uu))
                self.g[k] += (geq - self.g[k]) / tg + (1 - 0.5 / tg) * G
            for i in range(n):
                ti = self.p["tau"][i]
                R = (1 - 0.5 / ti) * 3 * self.w[k] * sum(c[d] * jump[i][d] for d in range(D))
                self.h[i, k] += (self.heq(k, i, ph[i], C[i], cu) - self.h[i, k]) / ti + R
        self.g, self.h = self.stream(self.g), self.stream(self.h)
        self.pp, self.up = ph, u

    def stream(self, f):
        """Push along c_k; halfway bounce-back at the walls. Directions lie before the grid's axes."""
        q = f.dim() - self.D - 1
        new = torch.empty_like(f)
        for k, c in enumerate(self.c):
            to, src = new.select(q, k), f.select(q, k)
            dims = [-1 - d for d in range(self.D) if c[d]]
            to.copy_(torch.roll(src, [c[d] for d in range(self.D) if c[d]], dims) if dims else src)
            if self.wall and c[1]:
                row = 0 if c[1] > 0 else f.shape[-2] - 1
                to.select(-2, row).copy_(f.select(q, self.opp[k]).select(-2, row))
        return new


def _simulate(p, c, u, steps):
    m = _Model(p)
    m.start(c, u)
    for _ in range(steps):
        m.step()
    return m.fields()


def exact(case, seed):
    rng = np.random.default_rng(seed)
    if case["kind"] == "batch":
        out = []
        for g, p, c, u in _batch_grids(case, rng):
            ph, _, _, _, _, _, _, v, _, pr = _simulate(p, c, u, case["steps"])
            out.append(torch.cat([ph, v, pr[None]]))
        return out
    p = _params(case, rng)
    c, u = _start(case, rng)
    ph, cc, rho, _, _, _, _, v, uu, pr = _simulate(p, c, u, case["steps"])
    out = {"phi": ph, "c": cc, "u": v, "p": pr, "rho": rho}
    if case["start"]:
        out["mass"] = cc.flatten(1).sum(1).cpu().numpy()
        out["ke"] = float((0.5 * rho * uu).sum())
        out["umax"] = float(uu.max().sqrt())
    return out
