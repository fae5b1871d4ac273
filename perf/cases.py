"""The work a user of this package has it do, as cases to be timed and checked.

A case is one whole solve through the public entry points: the initial mole
fractions go in (``set_state``), a run of time steps is taken (``step``) and
the mole fractions and fluxes come out (``moments``), as the problem drivers
of ``scenarios.py`` do between two samples; a batch of independent solves
likewise; or a gradient of a misfit through ``autograd.simulate``, forward and
backward.  Solvers (the plan a program keeps) are made in ``prepare``.
"""

import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_1808_06787_gb300 import BatchSolver, Solver
from paper_1808_06787_gb300.autograd import RunSpec, simulate

Q_OF = {"D1Q3": 3, "D2Q4": 4, "D2Q5": 5, "D2Q9": 9, "D3Q6": 6, "D3Q7": 7, "D3Q15": 15}
DIM_OF = {"D1Q3": 1, "D2Q4": 2, "D2Q5": 2, "D2Q9": 2, "D3Q6": 3, "D3Q7": 3, "D3Q15": 3}
FACES = {"p": "periodic", "w": "noflux", "d": "dirichlet"}
SIZE = {"f32": 4, "f64": 8}


def _grid(name, lattice, n, nx, ny, nz, dtype, faces, steps, field, relax="magic", flux=True, gradient=False):
    return {"name": name, "kind": "grid", "lattice": lattice, "n": n, "nx": nx, "ny": ny, "nz": nz,
            "dtype": dtype, "faces": faces, "steps": steps, "field": field, "relax": relax,
            "flux": flux, "gradient": gradient}


def listed():
    return [
        # a quick look at a small channel: every call is short, launches count
        _grid("channel 48x40 f32", "D2Q5", 3, 48, 40, 1, "f32", "wwpppp", 20, "sine"),
        # the binary step between Dirichlet walls (Sec. 4.1), to its first printed time
        _grid("erf walls 240x40 f64", "D2Q5", 2, 240, 40, 1, "f64", "ddpppp", 200, "erf"),
        # the seeded sine workload of the benchmark, in double precision
        _grid("sine 128x128 f64", "D2Q5", 3, 128, 128, 1, "f64", "pppppp", 200, "sine"),
        # the ternary coupling problem (Sec. 4.2): one of its 200 samples, with
        # the flux and the local gradient
        _grid("coupling 200x200 f64", "D2Q5", 3, 200, 200, 1, "f64", "wwpppp", 1666, "coupling", gradient=True),
        # double precision in 3D on a ragged closed box, for a converged reference
        _grid("box 101x96x67 f64", "D3Q7", 3, 101, 96, 67, "f64", "wwwwww", 20, "bulb"),
        # the benchmark's headline: two bulbs in a closed tube
        _grid("tube 256^3 f32", "D3Q7", 3, 256, 256, 256, "f32", "wwwwww", 20, "bulb"),
        # a ragged tube on the full 3D lattice, single relaxation time
        _grid("tube 161x127x143 f32", "D3Q15", 3, 161, 127, 143, "f32", "wwwwpp", 20, "bulb", relax="srt"),
        # five species in a plane
        _grid("blobs 2048x2048 f32", "D2Q9", 5, 2048, 2048, 1, "f32", "pppppp", 20, "blobs"),
        # a plane of the benchmark's plane workloads, odd sides, only x wanted
        _grid("plane 4095x4097 f32", "D2Q5", 3, 4095, 4097, 1, "f32", "wwpppp", 20, "bulb", flux=False),
        # a long line (a diffusion tube at high resolution)
        _grid("line 10000019 f32", "D1Q3", 3, 10000019, 1, 1, "f32", "wwpppp", 20, "bulb"),
        # thousands of uneven solves of a parameter study
        {"name": "batch of 4096 f32", "kind": "batch", "lattice": "D2Q5", "n": 3, "count": 4096, "lo": 32,
         "hi": 256, "dtype": "f32", "steps": 20, "flux": False},
        # the gradient of a misfit with respect to D_ij and the initial field
        {"name": "gradient 512x512 f32", "kind": "gradient", "lattice": "D2Q5", "n": 3, "nx": 512, "ny": 512,
         "nz": 1, "dtype": "f32", "faces": "pppppp", "steps": 200, "field": "sine", "relax": "magic"},
    ]


def _spread(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi], odd ones as often as even ones."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    kind = rng.choice(["paper", "paper", "small", "plane", "plane", "volume", "volume", "line", "batch", "gradient"])
    if kind == "paper":  # the paper's problems at other resolutions, double precision
        field, n, faces = rng.choice([("erf", 2, "ddpppp"), ("coupling", 3, "wwpppp"), ("sine", 3, "pppppp"),
                                      ("loschmidt", 3, "ppwwpp")])
        nx, ny = _spread(rng, 40, 600), _spread(rng, 8, 600)
        return _unnamed(_grid("", "D2Q5", n, nx, ny, 1, "f64", faces, _spread(rng, 50, 1000), field,
                              relax=rng.choice(["magic", "magic", "srt"]), gradient=rng.random() < 0.5))
    if kind == "small":
        lattice = rng.choice(["D2Q5", "D2Q5", "D2Q9", "D1Q3", "D3Q7"])
        dim = DIM_OF[lattice]
        nx = _spread(rng, 16, 160 if dim < 3 else 40)
        ny = _spread(rng, 8, 160 if dim == 2 else 24) if dim > 1 else 1
        nz = _spread(rng, 4, 24) if dim > 2 else 1
        return _unnamed(_grid("", lattice, rng.choice([2, 3, 3, 4]), nx, ny, nz, rng.choice(["f32", "f32", "f64"]),
                              rng.choice(["pppppp", "wwpppp"]), _spread(rng, 10, 200), "sine"))
    if kind == "plane":
        lattice = rng.choice(["D2Q5", "D2Q5", "D2Q9", "D2Q4"])
        nx, ny = _spread(rng, 300, 4096), _spread(rng, 300, 4096)
        n = rng.choice([2, 3, 3, 5]) if lattice != "D2Q4" else 3
        return _unnamed(_grid("", lattice, n, nx, ny, 1, "f32", rng.choice(["pppppp", "wwpppp", "wwwwpp"]), 20,
                              rng.choice(["sine", "bulb", "blobs"]) if n > 2 else "sine",
                              relax=rng.choice(["magic", "magic", "srt"]), flux=rng.random() < 0.5))
    if kind == "volume":
        lattice = rng.choice(["D3Q7", "D3Q7", "D3Q6", "D3Q15"])
        top = 256 if lattice != "D3Q15" else 180
        nx, ny, nz = (_spread(rng, 48, top) for _ in range(3))
        dtype = rng.choice(["f32", "f32", "f32", "f64"])
        return _unnamed(_grid("", lattice, rng.choice([2, 3, 3]), nx, ny, nz, dtype,
                              rng.choice(["wwwwww", "wwwwpp", "pppppp"]), 20, "sine", flux=rng.random() < 0.5))
    if kind == "line":
        return _unnamed(_grid("", "D1Q3", rng.choice([2, 3]), _spread(rng, 1000, 20000000), 1, 1, "f32",
                              rng.choice(["wwpppp", "pppppp"]), 20, "sine"))
    if kind == "batch":
        hi = _spread(rng, 64, 256)
        return {"kind": "batch", "lattice": "D2Q5", "n": rng.choice([2, 3, 3]), "count": _spread(rng, 64, 3000),
                "lo": _spread(rng, 16, 64), "hi": hi, "dtype": "f32", "steps": _spread(rng, 10, 60), "flux": rng.random() < 0.5}
    side = _spread(rng, 64, 512)
    return {"kind": "gradient", "lattice": rng.choice(["D2Q5", "D2Q5", "D2Q9"]), "n": 3, "nx": side,
            "ny": _spread(rng, 64, 512), "nz": 1, "dtype": rng.choice(["f32", "f32", "f64"]),
            "faces": rng.choice(["pppppp", "wwpppp"]), "steps": _spread(rng, 16, 120), "field": "sine", "relax": "magic"}


def _unnamed(c):
    del c["name"]
    return c


# --- inputs ------------------------------------------------------------------

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _rng(seed):
    return np.random.Generator(np.random.PCG64(int(seed)))


def _dtype(case):
    return {"f32": torch.float32, "f64": torch.float64}[case["dtype"]]


def _diffusivities(n, g):
    """Lattice diffusivities: one pair at 0.1, the others in [0.01, 0.12]."""
    D = np.ones((n, n))
    for i in range(n):
        for j in range(i + 1, n):
            D[i, j] = D[j, i] = 0.1 if (i, j) == (0, 1) else g.uniform(0.01, 0.12)
    return D


def _field(case, g, walls):
    """Initial mole fractions [n, nz, ny, nx], float64, summing to one at every node."""
    n, nx, ny, nz = case["n"], case["nx"], case["ny"], case["nz"]
    dev = _device()
    X = ((torch.arange(nx, device=dev, dtype=torch.float64) + 0.5) / nx).view(1, 1, nx)
    Y = ((torch.arange(ny, device=dev, dtype=torch.float64) + 0.5) / ny).view(1, ny, 1)
    Z = ((torch.arange(nz, device=dev, dtype=torch.float64) + 0.5) / nz).view(nz, 1, 1)
    one = torch.ones(nz, ny, nx, device=dev, dtype=torch.float64)
    x = torch.empty(n, nz, ny, nx, device=dev, dtype=torch.float64)
    shift = float(g.uniform(-0.05, 0.05))
    if case["field"] == "erf":  # a step from C0 to C1
        x[0] = torch.where(X < 0.5 + shift, walls[0][0] * one, walls[1][0] * one)
        x[1] = 1.0 - x[0]
    elif case["field"] == "coupling":  # the profile of Sec. 4.2
        p = torch.where(X < 0.25, 0.8 * one, torch.clamp(1.6 * (0.75 - X), min=0.0) * one)
        x[0] = p * (1.0 + shift)
        x[1] = 0.2 * (1.0 - abs(shift))
        x[2] = 1.0 - x[0] - x[1]
    elif case["field"] == "loschmidt":  # the two gas mixtures of Sec. 4.3
        low, high = (0.0, 0.509 + 0.1 * shift, 0.491 - 0.1 * shift), (0.515, 0.485, 0.0)
        for s in range(3):
            x[s] = torch.where(Y < 0.5, low[s] * one, high[s] * one)
    elif case["field"] == "bulb":  # two compositions, a tanh interface four cells wide
        h = 0.5 * (1.0 + torch.tanh((X - 0.5 - shift) * nx / 4.0)) * one
        left = np.linspace(0.0, 1.0, n)
        left /= left.sum()
        for s in range(n):
            x[s] = left[s] + (left[n - 1 - s] - left[s]) * h
    elif case["field"] == "blobs":
        x[:] = 1.0 / n
        for s in range(n):
            for _ in range(8):
                cx, cy = g.uniform(0.0, 1.0, 2)
                dx, dy = (X - cx).abs(), (Y - cy).abs()
                dx, dy = torch.minimum(dx, 1.0 - dx) * nx, torch.minimum(dy, 1.0 - dy) * ny
                x[s] += 0.2 * torch.exp(-(dx * dx + dy * dy) / (2.0 * 32.0 ** 2))
    else:  # one Fourier mode per species
        for s in range(n):
            k = g.integers(1, 5, 3)
            arg = 2.0 * math.pi * (k[0] * X + (k[1] * Y if ny > 1 else 0.0) + (k[2] * Z if nz > 1 else 0.0))
            x[s] = 1.0 / n + 0.05 * torch.sin(arg + float(g.uniform(0.0, 2.0 * math.pi)))
    return x / x.sum(0, keepdim=True)


def _walls(case, g):
    """{face: composition} of the Dirichlet walls (Sec. 4.1: 0.9 and 0.1)."""
    if "d" not in case["faces"]:
        return {}
    e = float(g.uniform(-0.02, 0.02))
    return {0: (0.9 + e, 0.1 - e), 1: (0.1 + e, 0.9 - e)}


def _problem(case, seed):
    """(diffusivities, initial field of the case's dtype, wall compositions by face)"""
    g = _rng(seed)
    D = _diffusivities(case["n"], g)
    walls = _walls(case, g)
    return D, _field(case, g, walls).to(_dtype(case)).contiguous(), walls


def _sides(case):
    """The study's grid sides, uniform in [lo, hi]: part of the case, the same for every input."""
    return _rng(1004).integers(case["lo"], case["hi"] + 1, size=case["count"])


def _batch_problem(case, seed):
    """(sides, diffusivities, faces, packed field): even instances are periodic with a
    Fourier mode per species, odd ones a closed channel with a tanh interface."""
    g = _rng(seed)
    n, count = case["n"], case["count"]
    sides = _sides(case)
    Ds = np.stack([_diffusivities(n, g) for _ in range(count)])
    faces = ["pppppp" if i % 2 == 0 else "wwpppp" for i in range(count)]
    dev = _device()
    side = torch.from_numpy(sides).to(dev)
    cells = side * side
    inst = torch.repeat_interleave(torch.arange(count, device=dev), cells)
    start = torch.cumsum(cells, 0) - cells
    local = torch.arange(int(cells.sum()), device=dev) - start[inst]
    L = side[inst]
    X = (local % L + 0.5) / L
    Y = (torch.div(local, L, rounding_mode="floor") + 0.5) / L
    odd = (inst % 2).bool()
    h = 0.5 * (1.0 + torch.tanh((X - 0.5) * L / 4.0))
    left = np.linspace(0.0, 1.0, n)
    left /= left.sum()
    k = torch.from_numpy(g.integers(1, 5, size=(n, 2, count))).to(dev)
    phi = torch.from_numpy(g.uniform(0.0, 2.0 * math.pi, size=(n, count))).to(dev)
    xs = []
    for s in range(n):
        wave = 1.0 / n + 0.05 * torch.sin(2.0 * math.pi * (k[s, 0][inst] * X + k[s, 1][inst] * Y) + phi[s][inst])
        xs.append(torch.where(odd, left[s] + (left[n - 1 - s] - left[s]) * h, wave))
    tot = sum(xs)
    flat = torch.empty(n * int(cells.sum()), device=dev, dtype=_dtype(case))
    at = n * start[inst] + local  # instance blocks [n, side, side], one after the other
    for s in range(n):
        flat[at + s * cells[inst]] = (xs[s] / tot).to(_dtype(case))
    return sides, Ds, faces, flat


def prepare(case, seed):
    if case["kind"] == "batch":
        sides, Ds, faces, flat = _batch_problem(case, seed)
        b = BatchSolver(case["lattice"], Ds, [(int(v), int(v)) for v in sides], bcs=[[FACES[c] for c in f] for f in faces],
                        dtype=_dtype(case))
        return {"case": case, "solver": b, "x0": flat}
    D, x0, walls = _problem(case, seed)
    bc = [FACES[c] for c in case["faces"]]
    grid = (case["nx"], case["ny"], case["nz"])
    if case["kind"] == "gradient":
        target = _problem(case, seed + 7)[1]
        pairs = torch.tensor([D[i, j] for i in range(case["n"]) for j in range(i + 1, case["n"])], dtype=torch.float64)
        return {"case": case, "x0": x0, "pairs": pairs, "target": target, "grid": grid, "bc": bc}
    s = Solver(case["lattice"], D, grid, bc=bc, relax=case["relax"], dtype=_dtype(case), boundary=walls)
    return {"case": case, "solver": s, "x0": x0}


def run(state):
    case = state["case"]
    if case["kind"] == "gradient":
        x0 = state["x0"].detach().clone().requires_grad_(True)
        d = state["pairs"].detach().clone().requires_grad_(True)
        spec = RunSpec(case["lattice"], state["grid"], case["steps"], bc=state["bc"], relax=case["relax"],
                       dtype=_dtype(case))
        x = simulate(x0, d, spec)
        misfit = 0.5 * (x - state["target"]).square().sum()
        misfit.backward()
        return {"x": x.detach(), "grad_x0": x0.grad, "grad_D": d.grad}
    s = state["solver"]
    s.set_state(state["x0"])
    s.step(case["steps"])
    if case["flux"]:
        x, J = s.moments(flux=True)
        out = {"x": x, "J": J}
    else:
        out = {"x": s.moments()}
    if case.get("gradient"):
        out["G"] = s.gradient()
    return out


def _cells(case):
    if case["kind"] == "batch":
        return int((_sides(case) ** 2).sum())
    return case["nx"] * case["ny"] * case["nz"]


def work(case):
    """Bytes of the fields that go in and come out, and the operations of the steps:
    sums, relaxation matrices (Eqs. 2-10, 3-26, 3-16) and the collision of every
    opposite pair at every node."""
    cells, n, S, Q, dim = _cells(case), case["n"], case["n"] - 1, Q_OF[case["lattice"]], DIM_OF[case["lattice"]]
    es = SIZE[case["dtype"]]
    fields = 2 * n + (n * dim if case.get("flux") else 0) + (n * dim if case.get("gradient") else 0)
    matrices = 4 * S * S + 2 * S * S * S + 6 * S
    collision = (Q // 2) * (7 * S + 4 * S * S) + 4 * S
    flops = case["steps"] * cells * (S * Q + matrices + collision)
    if case["kind"] == "gradient":  # forward, the states again, and an adjoint step of about twice the forward's work
        fields += n
        flops *= 4
    return {"bytes": float(fields * cells * es), "flops": float(flops)}


# --- the model in 64 bits, in plain torch ---------------------------------------

def _velocities(lattice):
    """Velocities, weights and c_s^2 of Sec. 3.1 (c_s^2 = sum_k w_k c_kx^2)."""
    axes = [v for a in range(3) for v in (tuple(1 if b == a else 0 for b in range(3)), tuple(-1 if b == a else 0 for b in range(3)))]
    rest = [(0, 0, 0)]
    diag2 = [(a, b, 0) for a in (1, -1) for b in (1, -1)]
    diag3 = [(a, b, c) for a in (1, -1) for b in (1, -1) for c in (1, -1)]
    c, w = {
        "D1Q3": (rest + axes[:2], [2 / 3] + [1 / 6] * 2),
        "D2Q4": (axes[:4], [1 / 4] * 4),
        "D2Q5": (rest + axes[:4], [1 / 3] + [1 / 6] * 4),
        "D2Q9": (rest + axes[:4] + diag2, [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4),
        "D3Q6": (axes, [1 / 6] * 6),
        "D3Q7": (rest + axes, [1 / 4] + [1 / 8] * 6),
        "D3Q15": (rest + axes + diag3, [2 / 9] + [1 / 9] * 6 + [1 / 72] * 8),
    }[lattice]
    return c, w, sum(wk * ck[0] ** 2 for ck, wk in zip(c, w))


class _Model:
    """The scheme on a flat set of nodes: coordinates x, y, z in grids of extents ext
    (tensors or numbers), `first` the index of the grid's first node, `wall(axis, high)` the
    nodes' mask of wall faces, 1/D_ij as numbers or per-node tensors."""

    def __init__(self, lattice, n, inv_d, pos, ext, first, wall, walls, relax):
        self.n, self.S, self.inv_d, self.relax = n, n - 1, inv_d, relax
        self.c, self.w, self.cs2 = _velocities(lattice)
        self.opp = [self.c.index(tuple(-v for v in ck)) for ck in self.c]
        self.src, self.bounce, self.fixed = [], [], []
        here = first + pos[0] + ext[0] * (pos[1] + ext[1] * pos[2])
        for k, ck in enumerate(self.c):
            crossed = torch.zeros_like(here, dtype=torch.bool)
            fixed = None
            q = list(pos)
            for a in range(3):
                if ck[a] == 0:
                    continue
                q[a] = pos[a] - ck[a]
                out = (q[a] < 0) if ck[a] > 0 else (q[a] >= ext[a])
                hit = out & wall(a, ck[a] < 0)
                face = 2 * a + (0 if ck[a] > 0 else 1)
                if face in walls:
                    fixed = (hit & ~crossed, walls[face])
                crossed = crossed | hit
                q[a] = torch.remainder(q[a], ext[a])
            there = first + q[0] + ext[0] * (q[1] + ext[1] * q[2])
            self.src.append(torch.where(crossed, here, there))
            self.bounce.append(crossed if bool(crossed.any()) else None)
            self.fixed.append(fixed)

    def gather(self, f):
        """f[s][k] -> the propagated populations (half-way bounce-back, anti-bounce-back)."""
        out = []
        for s in range(self.S):
            row = []
            for k in range(len(self.c)):
                v = f[s][k][self.src[k]] if any(self.c[k]) else f[s][k]
                if self.bounce[k] is not None:
                    v = torch.where(self.bounce[k], f[s][self.opp[k]], v)
                if self.fixed[k] is not None:
                    mask, xb = self.fixed[k]
                    v = torch.where(mask, 2.0 * self.w[k] * xb[s] - f[s][self.opp[k]], v)
                row.append(v)
            out.append(row)
        return out

    def fractions(self, f):
        x = [sum(f[s][1:], f[s][0]) for s in range(self.S)]
        return x + [1.0 - sum(x[1:], x[0])]

    def matrices(self, x):
        """Lambda_1 = (B^-1 / c_s^2 + I/2)^-1 = (I / c_s^2 + B/2)^-1 B by elimination, and
        Lambda_2 (Eq. 3-16, or Lambda_1)."""
        S, n, c = self.S, self.n, self.inv_d
        B = [[None] * S for _ in range(S)]
        for i in range(S):
            for j in range(S):
                if i == j:
                    B[i][i] = x[i] * c[i][n - 1] + sum(x[k] * c[i][k] for k in range(n) if k != i)
                else:
                    B[i][j] = x[i] * (c[i][n - 1] - c[i][j])
        K = [[B[i][j] * 0.5 + (1.0 / self.cs2 if i == j else 0.0) for j in range(S)] for i in range(S)]
        R = [list(r) for r in B]
        for p in range(S):
            for r in range(S):
                if r == p:
                    continue
                m = K[r][p] / K[p][p]
                K[r] = [K[r][j] - m * K[p][j] for j in range(S)]
                R[r] = [R[r][j] - m * R[p][j] for j in range(S)]
        L1 = [[R[i][j] / K[i][i] for j in range(S)] for i in range(S)]
        if self.relax == "srt":
            return L1, L1
        L2 = [[8.0 * (L1[i][i] - 2.0) / (L1[i][i] - 8.0) if i == j else L1[i][j] for j in range(S)] for i in range(S)]
        return L1, L2

    def collide(self, f):
        x = self.fractions(f)
        L1, L2 = self.matrices(x)
        S = self.S
        out = [[None] * len(self.c) for _ in range(S)]
        for k, o in enumerate(self.opp):
            if o < k:
                continue
            even = [0.5 * (f[s][k] + f[s][o]) - self.w[k] * x[s] for s in range(S)]
            odd = [0.5 * (f[s][k] - f[s][o]) for s in range(S)]
            for i in range(S):
                e = sum(L2[i][j] * even[j] for j in range(S))
                if o == k:
                    out[i][k] = f[i][k] - e
                    continue
                a = sum(L1[i][j] * odd[j] for j in range(S))
                out[i][k], out[i][o] = f[i][k] - e - a, f[i][o] - e + a
        return out

    def start(self, x0):
        return [[wk * x0[s] for wk in self.w] for s in range(self.S)]

    def run(self, x0, steps):
        """(post-collision populations, propagated ones of the last step)"""
        f = self.start(x0)
        g = f
        for _ in range(steps):
            g = self.gather(f)
            f = self.collide(g)
        return f, g

    def flux(self, g, dim):
        """J = (I - Lambda_1/2) m_1 and grad x = -Lambda_1 m_1 / c_s^2, [n][dim]."""
        L1, _ = self.matrices(self.fractions(g))
        J, G = [], []
        m = [[sum(ck[a] * g[s][k] for k, ck in enumerate(self.c) if ck[a]) for a in range(dim)] for s in range(self.S)]
        for i in range(self.S):
            lm = [sum(L1[i][j] * m[j][a] for j in range(self.S)) for a in range(dim)]
            J.append([m[i][a] - 0.5 * lm[a] for a in range(dim)])
            G.append([-lm[a] / self.cs2 for a in range(dim)])
        J.append([-sum(J[i][a] for i in range(self.S)) for a in range(dim)])
        G.append([-sum(G[i][a] for i in range(self.S)) for a in range(dim)])
        return J, G


def _grid_model(case, D, walls, inv_d=None):
    nx, ny, nz, n = case["nx"], case["ny"], case["nz"], case["n"]
    at = torch.arange(nx * ny * nz, device=_device())
    pos = [at % nx, torch.div(at, nx, rounding_mode="floor") % ny, torch.div(at, nx * ny, rounding_mode="floor")]
    closed = [f != "p" for f in case["faces"]]
    wall = lambda a, high: closed[2 * a + (1 if high else 0)]  # noqa: E731
    c = inv_d or [[1.0 / D[i, j] for j in range(n)] for i in range(n)]
    return _Model(case["lattice"], n, c, pos, (nx, ny, nz), 0, wall, walls, case["relax"])


def exact(case, seed):
    n, dim = case["n"], DIM_OF[case["lattice"]]
    if case["kind"] == "batch":
        sides, Ds, faces, flat = _batch_problem(case, seed)
        dev = flat.device
        side = torch.from_numpy(sides).to(dev)
        cells = side * side
        inst = torch.repeat_interleave(torch.arange(len(sides), device=dev), cells)
        first = (torch.cumsum(cells, 0) - cells)[inst]
        local = torch.arange(int(cells.sum()), device=dev) - first
        L, size = side[inst], cells[inst]
        pos = [local % L, torch.div(local, L, rounding_mode="floor"), torch.zeros_like(local)]
        closed = torch.tensor([[ch != "p" for ch in f] for f in faces], device=dev)
        wall = lambda a, high: closed[:, 2 * a + (1 if high else 0)][inst]  # noqa: E731
        c = [[torch.from_numpy(1.0 / Ds[:, i, j]).to(dev)[inst] for j in range(n)] for i in range(n)]
        m = _Model(case["lattice"], n, c, pos, (L, L, 1), first, wall, {}, "magic")
        at = n * first + local
        f, g = m.run([flat[at + s * size].double() for s in range(n - 1)], case["steps"])
        x = torch.empty(flat.shape, device=dev, dtype=torch.float64)
        for s, v in enumerate(m.fractions(f)):
            x[at + s * size] = v
        if not case["flux"]:
            return {"x": x}
        J = torch.empty(flat.numel() * dim, device=dev, dtype=torch.float64)
        fl = m.flux(g, dim)[0]
        for s in range(n):
            for a in range(dim):
                J[n * dim * first + local + (s * dim + a) * size] = fl[s][a]
        return {"x": x, "J": J}
    D, x0, walls = _problem(case, seed)
    shape = (case["nz"], case["ny"], case["nx"])
    if case["kind"] == "gradient":
        target = _problem(case, seed + 7)[1].double()
        pairs = torch.tensor([D[i, j] for i in range(n) for j in range(i + 1, n)], dtype=torch.float64, device=x0.device,
                             requires_grad=True)
        inv, k = [[0.0] * n for _ in range(n)], 0
        for i in range(n):
            for j in range(i + 1, n):
                inv[i][j] = inv[j][i] = 1.0 / pairs[k]
                k += 1
        m = _grid_model(case, D, walls, inv)
        start = x0.double().reshape(n, -1).requires_grad_(True)
        Q = len(m.c)

        def segment(flat, count):
            f = [[flat[s * Q + k] for k in range(Q)] for s in range(n - 1)]
            for _ in range(count):
                f = m.collide(m.gather(f))
            return torch.stack([v for row in f for v in row])

        f = torch.stack([v for row in m.start(start) for v in row])
        left = case["steps"]
        while left > 0:
            f = torch.utils.checkpoint.checkpoint(segment, f, min(left, 8), use_reentrant=False)
            left -= 8
        x = torch.stack(m.fractions([[f[s * Q + k] for k in range(Q)] for s in range(n - 1)])).view((n,) + shape)
        (0.5 * (x - target).square().sum()).backward()
        return {"x": x.detach(), "grad_x0": start.grad.view((n,) + shape), "grad_D": pairs.grad.cpu()}
    m = _grid_model(case, D, walls)
    f, g = m.run(x0.double().reshape(n, -1), case["steps"])
    out = {"x": torch.stack(m.fractions(f)).view((n,) + shape)}
    if case["flux"] or case["gradient"]:
        J, G = m.flux(g, dim)
        if case["flux"]:
            out["J"] = torch.stack([v for r in J for v in r]).view((n, dim) + shape)
        if case["gradient"]:
            out["G"] = torch.stack([v for r in G for v in r]).view((n, dim) + shape)
    return out
