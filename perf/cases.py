"""The work of this library that is timed: solves, a time step, a batch and single operator calls.

Every case goes through the package's public entry points (`assemble_operator`, `Operator.solve`,
`Operator.solve_noalloc`, `Operator.residual`, `Operator.spmv`, `Batch.solve`, `project_step`). A
user's program keeps a basin's operator, its time-step state or its batch and calls these once per
right-hand side or per step, so that is what a state holds and what `run` does.

Basins are the shapes the library is used on: unit-square boxes of depth 0.01 (the small test box,
the batch and serving set) and layered ocean basins with coastlines, an island, seeded bathymetry,
the viscosity and the one-month time step of the 512 x 512 x 32 benchmark basin.

`exact` restates the discrete problem in plain torch, in 64 bits, on the full node grid: the P1
element integrals of the six tetrahedra of every cell summed into 15 offsets per node, and the
solutions by conjugate gradients to the limit of the arithmetic.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_1207_0486_gb300 as pm

SYSTEMS = {"u1": pm.OP_VEL_U1, "u2": pm.OP_VEL_U2, "u3": pm.OP_VEL_U3, "pressure": pm.OP_PRESSURE,
           "mass": pm.OP_MASS}
PRECS = {"jacobi": pm.PREC_JACOBI, "ic0": pm.PREC_IC0, "line": pm.PREC_LINE}
PRECISIONS = {"fp64": pm.FP64, "fp32": pm.FP32_REFINE, "bf16": pm.BF16_REFINE}

# Slip walls: every wall of a box; south and north of an ocean basin.
BOX_WALLS, OCEAN_WALLS = 1 | 2 | 4 | 8, 4 | 8


def solve_case(name, basin, nx, ny, nz, system, prec, precision, rtol):
    return {"name": name, "kind": "solve", "basin": basin, "nx": nx, "ny": ny, "nz": nz, "shape": 1207,
            "system": system, "prec": prec, "precision": precision, "rtol": rtol}


def listed():
    return [
        # The small test box: one velocity solve and one pressure solve, where latency is all.
        solve_case("box_small_u1_ic0", "box", 16, 16, 8, "u1", "ic0", "fp64", 1e-10),
        solve_case("box_small_pressure_line", "box", 37, 29, 11, "pressure", "line", "fp64", 1e-10),
        # A regional basin, ragged sizes: the velocity prediction, where an iteration's many short
        # kernels count.
        solve_case("ocean_regional_u2_ic0", "ocean", 117, 90, 19, "u2", "ic0", "fp64", 1e-10),
        # Pressure of a box of the serving set.
        solve_case("box_serving_pressure_line", "box", 125, 125, 20, "pressure", "line", "fp64", 1e-10),
        # The benchmark basin's grid: velocity prediction and consistent-mass correction.
        solve_case("ocean_512_u1_ic0", "ocean", 512, 512, 32, "u1", "ic0", "fp64", 1e-10),
        solve_case("ocean_512_mass_ic0", "ocean", 512, 512, 32, "mass", "ic0", "fp64", 1e-10),
        # A large box of 32 levels, refinement with FP32 operator values.
        solve_case("box_large_pressure_fp32", "box", 384, 384, 32, "pressure", "line", "fp32", 1e-10),
        # BF16 operator values, velocity of a mid-sized basin.
        solve_case("ocean_mid_u1_ic0_bf16", "ocean", 224, 241, 27, "u1", "ic0", "bf16", 1e-10),
        # The allocation-free solve, by the diagonal, near its row limit.
        {"name": "box_noalloc_u3_jacobi", "kind": "noalloc", "basin": "box", "nx": 150, "ny": 141, "nz": 24,
         "shape": 1207, "system": "u3", "prec": "jacobi", "precision": "fp64", "rtol": 1e-10},
        # The true residual of the benchmark basin's pressure, as a user checks a solution with it.
        {"name": "ocean_512_residual", "kind": "residual", "basin": "ocean", "nx": 512, "ny": 512, "nz": 32,
         "shape": 1207, "system": "pressure"},
        # One BDF2 step with wind and Coriolis, the unit of every time loop.
        {"name": "box_step", "kind": "step", "basin": "box", "nx": 96, "ny": 96, "nz": 32, "shape": 1207,
         "rtol": 1e-11},
        # Many basins at once, four systems each, FP32 refinement (the batch set's sizes and rule).
        {"name": "batch_fp32", "kind": "batch", "basins": 6, "smin": 48, "smax": 160, "nzmin": 8, "nzmax": 48,
         "shape": 1207, "prec": "line", "precision": "fp32", "rtol": 1e-11},
    ]


def log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "solve", "solve", "noalloc", "residual", "step", "batch"])
    shape = rng.randrange(1 << 20)
    if kind == "batch":
        smin = log_int(rng, 24, 64)
        return {"kind": "batch", "basins": rng.randint(2, 6), "smin": smin, "smax": rng.randint(smin + 8, 150),
                "nzmin": 8, "nzmax": rng.randint(12, 48), "shape": shape, "prec": rng.choice(["line", "line", "ic0"]),
                "precision": rng.choice(["fp32", "fp32", "fp64", "bf16"]), "rtol": 1e-11}
    if kind == "step":
        side = log_int(rng, 14, 90)
        return {"kind": "step", "basin": "box", "nx": side, "ny": log_int(rng, 14, 90), "nz": rng.choice([8, 13, 20, 32]),
                "shape": shape, "rtol": 1e-11}
    basin = rng.choice(["box", "ocean"])
    nz = rng.choice([32, rng.randint(8, 48)])
    if kind == "noalloc":
        s = log_int(rng, 12, 100)
        return {"kind": kind, "basin": "box", "nx": s, "ny": log_int(rng, 12, 100), "nz": rng.randint(8, 32),
                "shape": shape, "system": rng.choice(["u1", "u3", "mass"]), "prec": "jacobi", "precision": "fp64",
                "rtol": 1e-10}
    if kind == "residual":
        return {"kind": kind, "basin": basin, "nx": log_int(rng, 48, 400), "ny": log_int(rng, 48, 400), "nz": nz,
                "shape": shape, "system": rng.choice(["u1", "u3", "pressure", "mass"])}
    system = rng.choice(["u1", "u2", "u3", "mass", "pressure"])
    prec = "line" if system == "pressure" else "ic0"
    if system == "pressure":
        basin = "box"
    lo, hi = (48, 400) if basin == "ocean" else (12, 320)
    nx = log_int(rng, lo, hi)
    ny = max(lo, min(hi, int(nx * rng.uniform(0.7, 1.4))))
    precision = rng.choice(["fp64", "fp64", "fp32", "bf16"]) if nx * ny * nz > 20000 else "fp64"
    return {"kind": "solve", "basin": basin, "nx": nx, "ny": ny, "nz": nz, "shape": shape, "system": system,
            "prec": prec, "precision": precision, "rtol": 1e-10}


# ---- inputs -------------------------------------------------------------------------------------

def box(nx, ny, nz):
    """The unit-square box of depth 0.01 with viscosity (1, 1, 1e-4)."""
    return SimpleNamespace(nx=nx, ny=ny, nz=nz, dx=1.0 / (nx - 1), dy=1.0 / (ny - 1), mask=np.ones((ny, nx), np.uint8),
                           depth=np.full((ny, nx), 0.01), slip_walls=BOX_WALLS, nu=(1.0, 1.0, 1e-4), dt=0.01,
                           coriolis=None)


def ocean(nx, ny, nz, shape):
    """A layered basin 5120 km across between two wavy coasts, with an island and seeded bathymetry."""
    rng = np.random.default_rng(shape)
    x = np.arange(nx)[None, :] / (nx - 1)
    y = np.arange(ny)[:, None] / (ny - 1)
    a, ph = rng.uniform(0.02, 0.05, 4), rng.uniform(0, 2 * math.pi, 4)
    west = 0.2 + a[0] * np.sin(2 * math.pi * y + ph[0]) + a[1] * np.sin(5 * math.pi * y + ph[1])
    east = 0.8 + a[2] * np.sin(2 * math.pi * y + ph[2]) + a[3] * np.sin(4 * math.pi * y + ph[3])
    cx, cy, rad = rng.uniform(0.42, 0.58), rng.uniform(0.3, 0.7), rng.uniform(0.04, 0.08)
    mask = (x >= west) & (x <= east) & ((x - cx) ** 2 + (y - cy) ** 2 > rad ** 2)
    g = np.zeros((ny, nx))
    for _ in range(40):
        gx, gy, w, h = rng.uniform(0, 1), rng.uniform(0, 1), rng.uniform(0.02, 0.15), rng.uniform(0.2, 1.0)
        g += h * np.exp(-((x - gx) ** 2) / (2 * w * w)) * np.exp(-((y - gy) ** 2) / (2 * w * w))
    g = (g - g.min()) / (g.max() - g.min())
    dx = 5.12e6 / nx
    coriolis = np.broadcast_to(2 * 7.2921e-5 * np.sin(np.deg2rad(70.0) * y), (ny, nx)).copy()
    return SimpleNamespace(nx=nx, ny=ny, nz=nz, dx=dx, dy=dx, mask=mask.astype(np.uint8), depth=200.0 + 4800.0 * g,
                           slip_walls=OCEAN_WALLS, nu=(1e8, 1e8, 1e2), dt=2.592e6, coriolis=coriolis)


def basin_of(case):
    if case["basin"] == "ocean":
        return ocean(case["nx"], case["ny"], case["nz"], case["shape"])
    b = box(case["nx"], case["ny"], case["nz"])
    if case["kind"] == "step":
        b.coriolis = np.broadcast_to(np.linspace(0.0, 1.0, b.ny)[:, None], (b.ny, b.nx)).copy()
    return b


def batch_of(case):
    """The batch set's rule: side log-uniform, depth levels uniform."""
    rng = np.random.default_rng(case["shape"])
    out = []
    for _ in range(case["basins"]):
        s = int(round(math.exp(rng.uniform(math.log(case["smin"]), math.log(case["smax"])))))
        out.append(box(s, s, int(rng.integers(case["nzmin"], case["nzmax"] + 1))))
    return out


def kept_columns(b):
    """Grid nodes of the kept columns: those with an ocean cell (four ocean corners) beside them."""
    m = b.mask.astype(bool)
    cell = m[:-1, :-1] & m[1:, :-1] & m[:-1, 1:] & m[1:, 1:]
    keep = np.zeros_like(m)
    for dj in (0, 1):
        for di in (0, 1):
            keep[dj:dj + cell.shape[0], di:di + cell.shape[1]] |= cell
    return cell, keep


def device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def grids(b):
    """x and y in [0, 1] and the depth fraction s (0 at the surface, 1 at the floor) of the kept
    columns' nodes, in the library's order (columns row by row, levels from the floor up)."""
    jj, ii = np.nonzero(kept_columns(b)[1])
    dev = device()
    x = torch.from_numpy(ii / (b.nx - 1)).to(dev)[:, None]
    y = torch.from_numpy(jj / (b.ny - 1)).to(dev)[:, None]
    s = 1.0 - torch.arange(b.nz, dtype=torch.float64, device=dev)[None, :] / (b.nz - 1)
    return x, y, s, torch.from_numpy(b.depth[jj, ii]).to(dev)[:, None]


def modes(gen, x, y, shapes=(torch.cos, torch.cos), count=4):
    """A seeded smooth horizontal field of `count` modes."""
    f = torch.zeros_like(x)
    for _ in range(count):
        a, m, l = float(torch.randn((), generator=gen)), int(torch.randint(1, 4, (), generator=gen)), \
            int(torch.randint(1, 4, (), generator=gen))
        f = f + a * shapes[0](m * math.pi * x) * shapes[1](l * math.pi * y)
    return f


def boundary(b):
    """The kept nodes of the (ny, nx, nz) grid, and per velocity component those with u = 0: coasts,
    closed outer walls, the floor, the normal component on slip walls, u3 at the surface."""
    dev, shape = device(), (b.ny, b.nx, b.nz)
    cell, keep = kept_columns(b)
    coast = torch.zeros(b.ny, b.nx, dtype=torch.bool, device=dev)
    pad = torch.ones(b.ny + 1, b.nx + 1, dtype=torch.bool, device=dev)
    pad[1:b.ny, 1:b.nx] = torch.from_numpy(cell).to(dev)
    for dj in (0, 1):
        for di in (0, 1):
            coast |= ~pad[dj:dj + b.ny, di:di + b.nx]
    wall = torch.zeros(2, b.ny, b.nx, dtype=torch.bool, device=dev)
    closed = torch.zeros_like(coast)
    for bit, axis, index in ((1, 0, (slice(None), 0)), (2, 0, (slice(None), -1)), (4, 1, (0,)), (8, 1, (-1,))):
        if b.slip_walls & bit:
            wall[axis][index] = True
        else:
            closed[index] = True
    floor = (coast | closed)[:, :, None].expand(shape).clone()
    floor[:, :, 0] = True
    fixed = [floor | wall[0][:, :, None], floor | wall[1][:, :, None], floor.clone()]
    fixed[2][:, :, -1] = True
    return torch.from_numpy(keep).to(dev)[:, :, None].expand(shape), fixed


def forcing(b, system, seed):
    """A right-hand side as a step makes it: a smooth body force and a surface-trapped wind drift, weighted
    by the nodes' volumes, with some small-scale content; a velocity's Dirichlet rows are 0."""
    gen = torch.Generator().manual_seed(seed)
    dgen = torch.Generator(device=device()).manual_seed(seed)
    x, y, s, h = grids(b)
    f = modes(gen, x, y) * (1.0 + 0.5 * torch.cos(math.pi * s)) + modes(gen, x, y) * torch.exp(-6.0 * s)
    f = f + 0.05 * torch.randn(f.shape, generator=dgen, device=f.device, dtype=f.dtype)
    f = f * h * (b.dx * b.dy / (b.nz - 1))
    f = f.reshape(-1)
    if system in ("u1", "u2", "u3"):
        keep, fixed = boundary(b)
        f[fixed[("u1", "u2", "u3").index(system)][keep]] = 0.0
    return f.contiguous()


def step_fields(b, seed):
    """u^k, u^{k-1}, p^k, the last pressure increment and the wind of a box in mid-run."""
    gen = torch.Generator().manual_seed(seed)
    x, y, s, _ = grids(b)
    sn = (torch.sin, torch.sin)
    up, bump = torch.sin(0.5 * math.pi * (1.0 - s)), torch.sin(math.pi * s)
    u = [(1e-2 * modes(gen, x, y, sn) * up).reshape(-1), (1e-2 * modes(gen, x, y, sn) * up).reshape(-1),
         (1e-4 * modes(gen, x, y, sn) * bump).reshape(-1)]
    prev = [0.97 * v for v in u]
    p = (1e-2 * modes(gen, x, y) + 0.0 * s).reshape(-1)
    q = 0.02 * p
    theta = [(-1e-4 * (1 + 0.1 * modes(gen, x, y)) * torch.cos(math.pi * y)).reshape(-1),
             (1e-5 * modes(gen, x, y)).reshape(-1)]
    return [v.contiguous() for v in u + prev + [p, q]], [t.contiguous() for t in theta]


def options(case):
    # the refinement of the single-system path restarts at 1e-2, that of a batch at 1e-4
    return pm.Options(rtol=case["rtol"], prec=PRECS[case["prec"]], precision=PRECISIONS[case["precision"]],
                      inner_rtol=1e-4 if case["kind"] == "batch" else 1e-2)


def batch_rhs(b, seed):
    """Seeded N(0, 1) right-hand sides of one basin's four systems (u1, u2, u3, pressure)."""
    gen = torch.Generator(device=device()).manual_seed(seed)
    n = b.nx * b.ny * b.nz
    return [torch.randn(n, generator=gen, device=device(), dtype=torch.float64) for _ in range(4)]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        basins = batch_of(case)
        ops = [pm.assemble_operator(b) for b in basins]
        bs = [v for k, b in enumerate(basins) for v in batch_rhs(b, seed * 64 + k)]
        which = [SYSTEMS[w] for _ in basins for w in ("u1", "u2", "u3", "pressure")]
        # "ic0": the velocities by IC0 and the pressure by its columns, mixed in one batch
        prec = [PRECS[case["prec"]]] * 3 + [pm.PREC_LINE]
        batch = pm.Batch([op for op in ops for _ in range(4)], which, options(case), prec=prec * len(basins))
        return SimpleNamespace(kind=kind, ops=ops, batch=batch, bs=bs, xs=[torch.zeros_like(b) for b in bs])
    b = basin_of(case)
    op = pm.assemble_operator(b)
    if kind == "step":
        fields, theta = step_fields(b, seed)
        return SimpleNamespace(kind=kind, op=op, st=pm.State(op), start=(fields, 5), theta=theta,
                               vel=pm.Options(rtol=case["rtol"], prec=pm.PREC_IC0),
                               pres=pm.Options(rtol=case["rtol"], prec=pm.PREC_LINE))
    rhs = forcing(b, case["system"], seed)
    s = SimpleNamespace(kind=kind, op=op, which=SYSTEMS[case["system"]], b=rhs, x=torch.zeros_like(rhs))
    if kind == "residual":
        s.x = forcing(b, case["system"], seed + (1 << 32))
        s.r = torch.empty_like(s.x)
    else:
        s.opts = options(case)
    return s


def run(state):
    s = state
    if s.kind == "solve":
        s.op.solve(s.which, s.b, s.x, s.opts)
        return s.x
    if s.kind == "noalloc":
        s.op.solve_noalloc(s.which, s.b, s.x, s.opts)
        return s.x
    if s.kind == "residual":
        norms = s.op.residual(s.which, s.b, s.x, s.r)
        return {"r": s.r, "norms": np.array(norms)}
    if s.kind == "batch":
        s.batch.solve(s.bs, s.xs)
        return s.xs
    s.st.restore(s.start)   # each pass is the same step of the time loop
    pm.project_step(s.op, s.st, s.theta[0], s.theta[1], s.vel, s.pres)
    return s.st.get()


# ---- the work a pass cannot do without -------------------------------------------------------------

def work(case):
    """Operator values, factors and vectors once each: a lower bound that no iteration count enters."""
    def rows(b):
        return int(kept_columns(b)[1].sum()) * b.nz
    if case["kind"] == "batch":
        n = sum(b.nx * b.ny * b.nz for b in batch_of(case))
        vb = {"fp64": 8, "fp32": 4, "bf16": 2}[case["precision"]]
        return {"bytes": n * (2 * 15 * vb + 15 * 8 + 4 * 16.0), "flops": n * 4 * 2 * 30.0}
    n = rows(basin_of(case))
    if case["kind"] == "step":
        return {"bytes": n * (2 * 15 * 8 + 8 * 8 + 4 * 8.0), "flops": n * 4 * 30.0 * 2}
    return {"bytes": n * (15 * 8 + 16.0 + (8 if case["kind"] == "residual" else 0)), "flops": n * 30.0}


# ---- the same problems in plain torch, in 64 bits ----------------------------------------------------

PERMS = ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0))


class Grid:
    """P1 operators on the full (ny, nx, nz) node grid; nodes of dropped columns have empty rows."""

    def __init__(self, b):
        dev = device()
        self.b, self.shape = b, (b.ny, b.nx, b.nz)
        cell, keep = kept_columns(b)
        self.cell = torch.from_numpy(cell).to(dev)
        self.keep = torch.from_numpy(keep).to(dev)[:, :, None].expand(self.shape)
        h = torch.from_numpy(b.depth).to(dev)
        self.z = -h[:, :, None] * (1.0 - torch.arange(b.nz, dtype=torch.float64, device=dev) / (b.nz - 1))
        self.fixed = boundary(b)[1]

    def tets(self):
        """For each of the six tetrahedra of every cell: the vertices' grid offsets, the volumes and the
        gradients of the four basis functions."""
        b = self.b
        ny, nx, nz = b.ny - 1, b.nx - 1, b.nz - 1
        live = self.cell[:, :, None].to(torch.float64)
        for p in PERMS:
            v = [[0, 0, 0]]
            for a in p:
                w = list(v[-1])
                w[a] += 1
                v.append(w)
            z = [self.z[o[1]:o[1] + ny, o[0]:o[0] + nx, o[2]:o[2] + nz] for o in v]
            # edge a of the path goes along axis p[a]: dz/d(edge) of each, and the three gradients
            dz = [z[k + 1] - z[k] for k in range(3)]
            step = [b.dx, b.dy, None]
            kz = p.index(2)
            inv_z = 1.0 / dz[kz]
            # mu_k: the coordinate along path edge k; lambda_0 = 1 - mu_0, lambda_k = mu_{k-1} - mu_k, lambda_3 = mu_2
            mu = [None] * 3
            zero, one = torch.zeros_like(inv_z), torch.ones_like(inv_z)
            for k in range(3):
                if k != kz:
                    mu[k] = [one / step[p[k]] if a == p[k] else zero for a in range(3)]
            mu[kz] = [zero, zero, inv_z]
            for k in range(3):
                if k != kz:
                    mu[kz][p[k]] = -(dz[k] / step[p[k]]) * inv_z
            grad = [[-mu[0][a] for a in range(3)], [mu[0][a] - mu[1][a] for a in range(3)],
                    [mu[1][a] - mu[2][a] for a in range(3)], mu[2]]
            yield v, live * (b.dx * b.dy * dz[kz].abs() / 6.0), grad

    def at(self, f, o):
        return f[o[1]:o[1] + self.b.ny - 1, o[0]:o[0] + self.b.nx - 1, o[2]:o[2] + self.b.nz - 1]

    def assemble(self, element):
        """Sum element(i, j, volume, gradients) into {offset: values at the row's node}."""
        A = {}
        for v, vol, grad in self.tets():
            for i in range(4):
                for j in range(4):
                    off = tuple(v[j][a] - v[i][a] for a in range(3))
                    if off not in A:
                        A[off] = torch.zeros(self.shape, dtype=torch.float64, device=self.z.device)
                    self.at(A[off], v[i]).add_(element(i, j, vol, grad))
        return A

    def operator(self, alpha, nu):
        """alpha M + K_nu (alpha = 0: K_nu; nu = 0: alpha M)."""
        def element(i, j, vol, grad):
            e = alpha * (2.0 if i == j else 1.0) / 20.0
            for a in range(3):
                if nu[a]:
                    e = e + nu[a] * grad[i][a] * grad[j][a]
            return vol * e
        return self.assemble(element)

    def system(self, name):
        """The eliminated operator of one system and its fixed nodes (None: none)."""
        if name == "pressure":
            return self.operator(0.0, (1.0, 1.0, 1.0)), None
        if name == "mass":
            return self.operator(1.0, (0.0, 0.0, 0.0)), None
        return self.operator(1.5 / self.b.dt, self.b.nu), self.fixed[("u1", "u2", "u3").index(name)]

    def apply(self, A, x):
        y = torch.zeros_like(x)
        for (di, dj, dk), a in A.items():
            src, dst = [], []
            for d, m in ((dj, self.shape[0]), (di, self.shape[1]), (dk, self.shape[2])):
                dst.append(slice(max(0, -d), m - max(0, d)))
                src.append(slice(max(0, d), m - max(0, -d)))
            y[tuple(dst)].addcmul_(a[tuple(dst)], x[tuple(src)])
        return y

    def spread(self, flat):
        """The library's vector (kept columns) on the full grid, and back."""
        f = torch.zeros(self.shape, dtype=torch.float64, device=self.z.device)
        f[self.keep] = flat
        return f

    def flat(self, f):
        return f[self.keep]

    def mass_sums(self):
        f = torch.zeros(self.shape, dtype=torch.float64, device=self.z.device)
        for v, vol, _ in self.tets():
            for i in range(4):
                self.at(f, v[i]).add_(vol / 4.0)
        return f

    def solve(self, name, rhs, limit=20000):
        """A x = rhs on the kept nodes, by conjugate gradients with each column's block as the
        preconditioner, restarted from the residual until that no longer falls."""
        A, fixed = self.system(name)
        free = self.keep if fixed is None else self.keep & ~fixed
        b = torch.where(self.keep, rhs, torch.zeros_like(rhs))
        x = torch.zeros_like(b)
        if fixed is not None:
            x = torch.where(self.keep & fixed, b, x)
            b = torch.where(free, b, torch.zeros_like(b))
        m = self.mass_sums() if name == "pressure" else None
        if m is not None:
            b = b - (b.sum() / m.sum()) * m
        off = lambda v: torch.where(free, v, torch.zeros_like(v))  # noqa: E731
        # the inverses of the columns' tridiagonal blocks
        d = torch.where(free, A[0, 0, 0], torch.ones_like(b))
        up = torch.where(free[:, :, :-1] & free[:, :, 1:], A[0, 0, 1][:, :, :-1], torch.zeros_like(b[:, :, 1:]))
        P = torch.linalg.inv(torch.diag_embed(d) + torch.diag_embed(up, 1) + torch.diag_embed(up, -1))

        def precondition(r):
            z = off((P @ r[..., None])[..., 0])
            return z if m is None else off(z - (m * z).sum() / m.sum())

        sol, r = torch.zeros_like(b), b
        best, size = math.inf, float(b.norm()) or 1.0
        for _ in range(8):
            e, q = torch.zeros_like(b), r.clone()
            z = precondition(q)
            p, rho = z, (q * z).sum()
            start = mark = float(q.norm())
            for it in range(limit):
                w = off(self.apply(A, p))
                alpha = rho / (p * w).sum()
                e += alpha * p
                q = q - alpha * w
                z = precondition(q)
                rho, old = (q * z).sum(), rho
                p = z + (rho / old) * p
                if it % 50 == 49 and not float(q.norm()) > 1e-7 * start:
                    break
                if it % 400 == 399:   # rounding keeps the residual from falling further
                    mark, last = float(q.norm()), mark
                    if not mark < 0.2 * last:
                        break
            trial = sol + e
            if m is not None:
                trial = off(trial - (m * trial).sum() / m.sum())
            r = off(b - self.apply(A, trial))
            now = float(r.norm())
            if now < best:
                sol = trial
            if not now < 0.3 * best or now < 1e-15 * size:
                break
            best = now
        return x + sol

    # ---- one time step -----------------------------------------------------------------------
    def gradients(self):
        return [self.assemble(lambda i, j, vol, grad, c=c: vol * grad[j][c] / 4.0) for c in range(3)]

    def velocity_rhs(self, u, prev, p, theta):
        b, dt = self.b, self.b.dt
        M = self.operator(1.0, (0.0, 0.0, 0.0))
        rhs = [self.apply(M, 2.0 * u[c] - 0.5 * prev[c]) / dt for c in range(3)]
        for v, vol, grad in self.tets():
            ul = [[self.at(u[c], v[i]) for i in range(4)] for c in range(3)]
            pl = sum(self.at(p, v[j]) for j in range(4))
            mu = [[vol * (sum(ul[d]) + ul[d][i]) / 20.0 for i in range(4)] for d in range(3)]
            for c in range(3):
                g = [sum(grad[j][d] * ul[c][j] for j in range(4)) for d in range(3)]
                for i in range(4):
                    self.at(rhs[c], v[i]).add_(vol * grad[i][c] / 4.0 * pl - sum(g[d] * mu[d][i] for d in range(3)))
        f = torch.from_numpy(b.coriolis).to(self.z.device)[:, :, None]
        rhs[0] += f * self.apply(M, u[1])
        rhs[1] -= f * self.apply(M, u[0])
        ny, nx = b.ny - 1, b.nx - 1
        live = self.cell.to(torch.float64)
        for corners in (((0, 0), (1, 0), (1, 1)), ((0, 0), (0, 1), (1, 1))):   # surface triangles
            for c in range(2):
                t = [theta[c][j:j + ny, i:i + nx] for i, j in corners]
                for k, (i, j) in enumerate(corners):
                    rhs[c][j:j + ny, i:i + nx, -1].add_(live * b.dx * b.dy / 24.0 * (sum(t) + t[k]))
        return [torch.where(self.fixed[c] | ~self.keep, torch.zeros_like(rhs[c]), rhs[c]) for c in range(3)]

    def step(self, fields, theta):
        v = [self.spread(f) for f in fields]
        u, prev, p = v[0:3], v[3:6], v[6]
        th = []
        for t in theta:
            g = torch.zeros(self.shape[:2], dtype=torch.float64, device=self.z.device)
            g[self.keep[:, :, 0]] = t
            th.append(g)
        alpha = 1.5 / self.b.dt
        rhs = self.velocity_rhs(u, prev, p, th)
        ut = [self.solve(name, rhs[c]) for c, name in enumerate(("u1", "u2", "u3"))]
        G = self.gradients()
        q = self.solve("pressure", -alpha * sum(self.apply(G[c], ut[c]) for c in range(3)))
        m = torch.where(self.keep, self.mass_sums(), torch.ones_like(p))
        new = [torch.where(self.fixed[c], torch.zeros_like(p), ut[c] - self.apply(G[c], q) / (alpha * m))
               for c in range(3)]
        return [self.flat(f) for f in new + [p + q]]


def exact(case, seed):
    if case["kind"] == "batch":
        out = []
        for k, b in enumerate(batch_of(case)):
            g = Grid(b)
            for name, rhs in zip(("u1", "u2", "u3", "pressure"), batch_rhs(b, seed * 64 + k)):
                out.append(g.flat(g.solve(name, g.spread(rhs))))
        return out
    b = basin_of(case)
    g = Grid(b)
    if case["kind"] == "step":
        return g.step(*step_fields(b, seed))
    rhs = g.spread(forcing(b, case["system"], seed))
    if case["kind"] == "residual":
        A, fixed = g.system(case["system"])
        x = g.spread(forcing(b, case["system"], seed + (1 << 32)))
        free = g.keep if fixed is None else g.keep & ~fixed
        y = torch.where(free, g.apply(A, torch.where(free, x, torch.zeros_like(x))), x)
        r = g.flat(rhs - y)
        return {"r": r, "norms": None}
    return g.flat(g.solve(case["system"], rhs))
