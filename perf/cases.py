"""The calls whose speed counts: what users of this library have it do, through
its public entry points (the C ABI by its ctypes binding, and the autograd
wrapper), over the sizes, precisions and options they use.

    listed()             the named cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  inputs on the GPU and the handle a program keeps
    run(state)           one pass: the call, and its outputs
    work(case)           bytes and operations a pass cannot do without
    exact(case, seed)    the same outputs in 64 bits, in plain torch

A run of a problem is set_state from a device tensor, step, get_state into a
device tensor, as a program does that starts from its own data and reads the
solution back.  Sizes: the meshes of the paper's tables and shock tests
(1D 40-800 cells, 2D 30-240 a side), the benchmark's grids (1D 65536, the
512-instance batch of 256-16384 cells, 2D 4096 x 4096, the adjoint), and what
lies between them, odd and ragged sizes included.
"""

import math
import random

import numpy as np
import torch

from paper_2002_08816_gb300 import hweno as H
from paper_2002_08816_gb300.autograd import HwenoRun2D

DEVICE = "cuda" if torch.cuda.is_available() else "cpu"
GAS = 1.4
EPS = 1e-6
PRECISION = {"fp32": H.HWENO_FP32, "fp64": H.HWENO_FP64, "fp32c": H.HWENO_FP32C}
BC = {"periodic": H.HWENO_BC_PERIODIC, "outflow": H.HWENO_BC_OUTFLOW,
      "reflective": H.HWENO_BC_REFLECTIVE}

# Operations per cell and Runge-Kutta stage of the scheme on smooth data, as
# counted on a plain implementation: (system, dimension, Gauss points).
FLOPS = {("euler", 1, 0): 544, ("burgers", 1, 0): 166, ("euler", 2, 2): 2898,
         ("euler", 2, 3): 4911, ("burgers", 2, 2): 675, ("burgers", 2, 3): 1137}


# ------------------------------------------------------------------ the cases

def _run1d(name, **kw):
    case = {"name": name, "kind": "run1d", "system": "euler", "data": "two_state", "bc": "outflow",
            "precision": "fp32", "threads": 0, "launch": 0, "cfl": 0.5}
    case.update(kw)
    return case


def _run2d(name, **kw):
    case = {"name": name, "kind": "run2d", "system": "euler", "data": "vortex", "bc": "periodic",
            "precision": "fp32", "gauss": 3, "cfl": 0.4}
    case.update(kw)
    return case


def listed():
    return [
        # a program's own time integrator, which calls the operator once per
        # stage on a paper-sized mesh: the smallest call, latency only
        {"name": "rhs1d_200_fp64", "kind": "rhs1d", "system": "euler", "data": "lax",
         "bc": "outflow", "precision": "fp64", "nx": 200, "cfl": 0.6},
        # the paper's Lax shock tube on its mesh, a handle as it is created
        _run1d("run1d_lax_200_fp32", data="lax", nx=200, steps=60, cfl=0.6),
        # a paper-sized shock problem in 64 bits, as its tables are computed
        _run1d("run1d_400_fp64", nx=400, steps=60, precision="fp64"),
        # the benchmark's 1D grid on the launch the README's autotuner picks
        _run1d("run1d_65536_fp32", nx=65536, steps=200, threads=256, launch=2),
        # the same grid with float-pair averages, for converged first moments
        _run1d("run1d_65536_fp32c", nx=65536, steps=100, precision="fp32c"),
        # the same grid in 64 bits
        _run1d("run1d_65536_fp64", nx=65536, steps=10, precision="fp64", threads=128, launch=1),
        # the benchmark's batch: an ensemble of uneven problems in one handle
        {"name": "batch1d_512_fp32", "kind": "batch1d", "system": "euler", "data": "two_state",
         "bc": "outflow", "precision": "fp32", "n_batch": 512, "lo": 256, "hi": 16384,
         "size_seed": 77, "steps": 12, "threads": 128, "launch": 0, "cfl": 0.5},
        # a parameter sweep of paper-sized meshes, the handle as it is created
        {"name": "batch1d_sweep_fp32", "kind": "batch1d", "system": "euler", "data": "lax",
         "bc": "outflow", "precision": "fp32", "n_batch": 250, "lo": 40, "hi": 800,
         "size_seed": 5, "steps": 16, "threads": 0, "launch": 0, "cfl": 0.5},
        # a paper-sized 2D mesh: fewer tiles than SMs
        _run2d("run2d_120_fp32", nx=120, ny=120, steps=30),
        # the benchmark's 2D grid
        _run2d("run2d_4096_fp32", nx=4096, ny=4096, gauss=2, steps=4),
        # a ragged 2D grid with shocks and open boundaries, in 64 bits
        _run2d("run2d_250x190_fp64", nx=250, ny=190, data="quadrants", bc="outflow",
               precision="fp64", steps=5),
        # the gradient of a loss through a recorded run (forward and backward)
        {"name": "adjoint2d_512_fp32", "kind": "adjoint2d", "system": "euler", "data": "vortex",
         "bc": "periodic", "precision": "fp32", "nx": 512, "ny": 512, "gauss": 3, "cfl": 0.4,
         "steps": 12, "every": 5},
    ]


def _unnamed(case):
    return {k: v for k, v in case.items() if k != "name"}


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run1d", "run1d", "run1d", "batch1d", "run2d", "run2d", "rhs1d", "rhs2d",
                       "adjoint2d"])
    if kind == "rhs1d":
        # 32 bits only where a jump and not the rounding sets the size of L
        precision = rng.choice(["fp64", "fp64", "fp32"])
        nx = _log(rng, 40, 100000) if precision == "fp64" else _log(rng, 40, 1000)
        return {"kind": kind, "system": "euler", "data": rng.choice(["lax", "two_state"]),
                "bc": rng.choice(["outflow", "periodic"]), "precision": precision, "nx": nx,
                "cfl": 0.6}
    if kind == "rhs2d":
        nx, ny = _log(rng, 30, 1024), _log(rng, 30, 1024)
        return {"kind": kind, "system": "euler", "data": "quadrants",
                "bc": rng.choice(["outflow", "periodic"]), "precision": "fp64", "nx": nx,
                "ny": ny, "gauss": rng.choice([2, 3]), "cfl": 0.4}
    if kind == "run1d":
        system, data, bc = rng.choice([("euler", "two_state", "outflow"), ("euler", "lax", "outflow"),
                                       ("euler", "two_state", "reflective"),
                                       ("euler", "wave", "periodic"),
                                       ("burgers", "burgers", "periodic")])
        precision = rng.choice(["fp32", "fp32", "fp64", "fp32c"])
        nx = _log(rng, 40, {"fp32": 1000000, "fp64": 100000, "fp32c": 65536}[precision])
        # the launches a program may choose by hand where the grid allows them
        # (the resident one needs 32 bits and all tiles on the GPU at once)
        choices = [(0, 0), (0, 0), (128, 0), (256, 1)]
        if precision == "fp32" and nx <= 65536:
            choices = [(0, 0), (0, 0), (128, 0), (256, 2)]
        threads, launch = (0, 0) if precision == "fp32c" else rng.choice(choices)
        cells = 4000000 if precision != "fp64" else 400000
        steps = max(4, min(120, cells // nx))
        return _unnamed(_run1d("", system=system, data=data, bc=bc, precision=precision, nx=nx,
                               threads=threads, launch=launch, steps=steps))
    if kind == "batch1d":
        lo, hi = rng.choice([(40, 800), (40, 1500), (256, 16384)])
        precision = rng.choice(["fp32", "fp32", "fp64"])
        # (many coarse shock problems at once hold cells at the very threshold of
        # the troubled-cell indicator, which 32 bits decide by their rounding)
        n_batch = _log(rng, 16, 1000 if precision == "fp64" and hi < 2000 else 400)
        threads, launch = rng.choice([(0, 0), (128, 0)])
        return {"kind": kind, "system": "euler", "data": "two_state" if lo > 40 else "lax",
                "bc": "outflow", "precision": precision, "n_batch": n_batch, "lo": lo, "hi": hi,
                "size_seed": rng.randrange(1000), "steps": 10 if precision == "fp32" else 4,
                "threads": threads, "launch": launch, "cfl": 0.5}
    if kind == "run2d":
        system, data, bc = rng.choice([("euler", "vortex", "periodic"), ("euler", "vortex", "periodic"),
                                       ("euler", "quadrants", "outflow"),
                                       ("burgers", "burgers", "periodic")])
        precision = rng.choice(["fp32", "fp32", "fp32c", "fp64"])
        top = 2048 if precision != "fp64" else 400
        nx = _log(rng, 30, top)
        ny = max(30, min(top, int(nx * rng.uniform(0.5, 2.0))))
        cells = 4000000 if precision != "fp64" else 200000
        steps = max(2, min(12 if data == "quadrants" else 40, cells // (nx * ny)))
        return _unnamed(_run2d("", system=system, data=data, bc=bc, precision=precision, nx=nx, ny=ny,
                               gauss=rng.choice([2, 3]), steps=steps))
    nx = _log(rng, 30, 600)
    ny = max(30, min(600, int(nx * rng.uniform(0.5, 2.0))))
    return {"kind": kind, "system": "euler", "data": "vortex", "bc": "periodic",
            "precision": rng.choice(["fp32", "fp32", "fp64"]) if nx * ny < 40000 else "fp32",
            "nx": nx, "ny": ny, "gauss": rng.choice([2, 3]), "cfl": 0.4,
            "steps": rng.choice([6, 12]), "every": rng.choice([3, 5, 20])}


# ------------------------------------------------------------ the initial data
# Point functions of the paper's problems (shock tubes, density waves, the
# isentropic vortex, four quadrants), with the seed's states, amplitudes and
# phases, turned into moments by Gauss quadrature on the device.

def _batch_sizes(case):
    if case["kind"] != "batch1d":
        return [case["nx"]]
    r = random.Random(case["size_seed"])
    return [_log(r, case["lo"], case["hi"]) for _ in range(case["n_batch"])]


def _gauss(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return 0.5 * x, 0.5 * w  # on [-1/2, 1/2], weights summing to 1


def _domain(case):
    """x0, x1, y0, y1; square cells in 2D."""
    if case["kind"].endswith("1d"):
        return (-1.0, 1.0, 0.0, 1.0) if case["data"] == "burgers" else (0.0, 1.0, 0.0, 1.0)
    side = {"burgers": 4.0, "vortex": 10.0, "quadrants": 10.0}[case["data"]]
    h = side / max(case["nx"], case["ny"])
    return 0.0, h * case["nx"], 0.0, h * case["ny"]


def _points1d(case, r, n):
    """f(x) -> [C, ...] for one problem of n cells."""
    data = case["data"]

    def conserved(rho, mu, p):
        return torch.stack([rho, rho * mu, p / (GAS - 1.0) + 0.5 * rho * mu * mu])

    if data == "burgers":
        a, c, k = 0.5 + 0.1 * r.random(), 0.8 + 0.4 * r.random(), r.random()
        return lambda x: (a + c * torch.sin(math.pi * x + 2.0 * math.pi * k))[None]
    if data == "wave":
        a, k = 0.1 + 0.2 * r.random(), r.random()
        return lambda x: conserved(1.0 + a * torch.sin(2.0 * math.pi * (x + k)),
                                   torch.ones_like(x), torch.ones_like(x))
    if data == "lax":
        s = [v * (1.0 + 0.05 * (2.0 * r.random() - 1.0)) for v in (0.445, 0.698, 3.528, 0.5, 0.571)]

        def lax(x):
            left = x < 0.5
            return conserved(torch.where(left, s[0], s[3]), torch.where(left, s[1], 0.0),
                             torch.where(left, s[2], s[4]))
        return lambda x: lax(x).to(torch.float64)
    # between walls the gas is nearly at rest (the paper's blast waves), so that
    # no wall starts with a vacuum beside it
    v = 0.1 if case["bc"] == "reflective" else 1.0
    left = (r.uniform(0.1, 1.0), r.uniform(-v, v), r.uniform(0.1, 1.0))
    right = (r.uniform(0.1, 1.0), r.uniform(-v, v), r.uniform(0.1, 1.0))
    top = max(1, min(256, n // 64))  # resolved on the coarsest mesh
    modes = [(r.randint(min(4, top), top), r.uniform(0.0, 2.0 * math.pi)) for _ in range(4)]

    def two_state(x):
        is_left = x < 0.5
        m = sum(torch.sin(2.0 * math.pi * k * x + ph) for k, ph in modes) / 4.0
        rho = torch.where(is_left, left[0], right[0] * (1.0 + 0.2 * m))
        mu = torch.where(is_left, left[1], right[1]).to(torch.float64)
        p = torch.where(is_left, left[2], right[2]).to(torch.float64)
        return conserved(rho, mu, p)
    return two_state


def _initial1d(case, seed):
    """The state in 64 bits: the instances' [C][2][n] one after the other."""
    x0, x1, _, _ = _domain(case)
    xi, w = _gauss(5)
    xi_d = torch.tensor(xi, device=DEVICE)[:, None]
    w_d = torch.tensor(w, device=DEVICE)
    parts = []
    for b, n in enumerate(_batch_sizes(case)):
        f = _points1d(case, random.Random(seed * 4099 + b), n)
        dx = (x1 - x0) / n
        x = x0 + (torch.arange(n, device=DEVICE, dtype=torch.float64) + 0.5) * dx
        v = f(x[None, :] + xi_d * dx)  # [C, points, n]
        avg = torch.einsum("q,cqn->cn", w_d, v)
        mom = torch.einsum("q,cqn->cn", w_d * xi_d[:, 0], v)
        parts.append(torch.stack([avg, mom], dim=1).reshape(-1))
    u = torch.cat(parts)
    return u if case["kind"] == "batch1d" else u.reshape(-1, 2, case["nx"])


def _points2d(case, r):
    x0, x1, y0, y1 = _domain(case)
    if case["data"] == "burgers":
        a, k = 0.4 + 0.2 * r.random(), r.random()
        lx, ly = x1 - x0, y1 - y0
        return lambda x, y: (a + torch.sin(2.0 * math.pi * (x / lx + y / ly + k)))[None]

    def conserved(rho, mu, nu, p):
        return torch.stack([rho, rho * mu, rho * nu, p / (GAS - 1.0) + 0.5 * rho * (mu * mu + nu * nu)])

    xm, ym = 0.5 * (x0 + x1), 0.5 * (y0 + y1)
    if case["data"] == "quadrants":
        st = [(r.uniform(0.3, 1.0), r.uniform(-0.8, 0.8), r.uniform(-0.8, 0.8), r.uniform(0.3, 1.0))
              for _ in range(4)]

        def quadrants(x, y):
            q = (x >= xm).long() + 2 * (y >= ym).long()
            return conserved(*[torch.tensor([s[k] for s in st], device=DEVICE, dtype=torch.float64)[q]
                               for k in range(4)])
        return quadrants
    top = max(2, min(16, min(case["nx"], case["ny"]) // 16))
    modes = [(r.randint(1, top), r.randint(1, top), r.uniform(0.0, 2.0 * math.pi)) for _ in range(8)]
    strength = 4.0 + 2.0 * r.random()

    def vortex(x, y):
        xb, yb = x - xm, y - ym
        r2 = xb * xb + yb * yb
        e = strength / (2.0 * math.pi) * torch.exp(0.5 * (1.0 - r2))
        temp = 1.0 - (GAS - 1.0) * strength ** 2 / (8.0 * GAS * math.pi ** 2) * torch.exp(1.0 - r2)
        rho = temp ** (1.0 / (GAS - 1.0))
        p = rho ** GAS
        m = sum(torch.sin(2.0 * math.pi * (a * (x - x0) / (x1 - x0) + b * (y - y0) / (y1 - y0)) + ph)
                for a, b, ph in modes) / len(modes)
        return conserved(rho * (1.0 + 0.05 * m), 1.0 - e * yb, 1.0 + e * xb, p)
    return vortex


def _initial2d(case, seed):
    x0, x1, y0, y1 = _domain(case)
    nx, ny = case["nx"], case["ny"]
    dx, dy = (x1 - x0) / nx, (y1 - y0) / ny
    f = _points2d(case, random.Random(seed * 4099 + 1))
    xi, w = _gauss(2 if nx * ny > 1 << 22 else 3)
    xc = x0 + (torch.arange(nx, device=DEVICE, dtype=torch.float64) + 0.5) * dx
    yc = y0 + (torch.arange(ny, device=DEVICE, dtype=torch.float64) + 0.5) * dy
    out = 0.0
    for a in range(len(w)):
        for b in range(len(w)):
            x, y = torch.broadcast_tensors((xc + xi[a] * dx)[None, :], (yc + xi[b] * dy)[:, None])
            v = f(x, y) * (w[a] * w[b])
            out = out + torch.stack([v, xi[a] * v, xi[b] * v], dim=1)
    return out


def _initial(case, seed):
    """The state a pass starts from, rounded to what the call is given."""
    u = _initial1d(case, seed) if case["kind"].endswith("1d") else _initial2d(case, seed)
    return u.to(torch.float32) if case["precision"] == "fp32" else u


# --------------------------------------------------------------- a user's calls

class _Handle:
    """A library handle that is destroyed with its owner."""

    def __init__(self, value):
        self.value = value

    def __del__(self):
        try:
            H.hweno_destroy(self.value)
        except Exception:
            pass


def _config(case):
    x0, x1, y0, y1 = _domain(case)
    system = H.HWENO_EULER if case["system"] == "euler" else H.HWENO_BURGERS
    if case["kind"].endswith("1d"):
        return H.make_config(1, system, case.get("nx", 4), x0=x0, x1=x1, bc=BC[case["bc"]],
                             cfl=case["cfl"], precision=PRECISION[case["precision"]])
    return H.make_config(2, system, case["nx"], case["ny"], x0=x0, x1=x1, y0=y0, y1=y1,
                         bc=BC[case["bc"]], cfl=case["cfl"], n_gauss=case["gauss"],
                         precision=PRECISION[case["precision"]])


def prepare(case, seed):
    u0 = _initial(case, seed).contiguous()
    state = {"case": case, "u0": u0, "out": torch.empty_like(u0)}
    cfg = _config(case)
    stream = torch.cuda.current_stream().cuda_stream
    if case["kind"] == "adjoint2d":
        state["u0"] = u0.requires_grad_(True)
        state["run"] = HwenoRun2D(cfg)
        return state
    if case["kind"] == "batch1d":
        state["sizes"] = _batch_sizes(case)
        state["handle"] = _Handle(H.hweno_create_batch(cfg, state["sizes"], stream))
    else:
        state["handle"] = _Handle(H.hweno_create(cfg, stream))
    if case.get("threads"):
        H.hweno_set_execution(state["handle"].value, case["threads"], case["launch"])
    if case["kind"].startswith("rhs"):
        state["ulim"] = torch.empty_like(u0)
        state["flags"] = torch.empty(u0.shape[2:], dtype=torch.uint8, device=DEVICE)
    return state


def run(state):
    case, u0, out = state["case"], state["u0"], state["out"]
    if case["kind"] == "adjoint2d":
        u = state["run"](u0, case["steps"], case["every"])
        grad, = torch.autograd.grad((u[0, 0] ** 2).sum(), u0)
        return {"state": u.detach(), "grad": grad}
    h = state["handle"].value
    if case["kind"].startswith("rhs"):
        H.hweno_rhs(h, u0.data_ptr(), out.data_ptr(), state["flags"].data_ptr(),
                    state["ulim"].data_ptr())
        return {"rhs": out, "ulim": state["ulim"], "flags": state["flags"]}
    # float-pair handles take and give 64-bit states, which hold the pairs
    dtype = H.HWENO_FP32 if u0.dtype == torch.float32 else H.HWENO_FP64
    H.hweno_set_state(h, u0.data_ptr(), dtype, True)
    t = H.hweno_step(h, case["steps"])
    H.hweno_get_state(h, out.data_ptr(), dtype, True)
    if case["kind"] == "batch1d":
        times = np.asarray(H.hweno_batch_times(h, len(state["sizes"])), dtype=np.float32)
        return {"state": out, "times": times}
    if case["precision"] == "fp32c":  # its averages are held to 2^-48, its moments to 2^-24
        return {"state": out.to(torch.float32), "t": t}
    return {"state": out, "t": t}


def work(case):
    dim = 1 if case["kind"].endswith("1d") else 2
    cells = sum(_batch_sizes(case)) if dim == 1 else case["nx"] * case["ny"]
    comps = {("burgers", 1): 1, ("euler", 1): 3, ("burgers", 2): 1, ("euler", 2): 4}[(case["system"], dim)]
    size = comps * (dim + 1) * (8 if case["precision"] == "fp64" else 4)
    flops = FLOPS[(case["system"], dim, case.get("gauss", 0))]
    if case["kind"].startswith("rhs"):  # the state in; L, the limited state and the flags out
        return {"bytes": cells * (3.0 * size + 1.0), "flops": float(cells) * flops}
    total = float(cells) * 3 * case["steps"] * flops
    if case["kind"] == "adjoint2d":  # state and gradient, in and out; forward and transposed
        return {"bytes": 4.0 * cells * size, "flops": 3.0 * total}
    return {"bytes": 2.0 * cells * size, "flops": total}


# ------------------------------------------------------------- the same in 64 bits
# The scheme in plain torch: every candidate polynomial solved from its moment
# conditions in the reference cell [-1/2, 1/2]^d, every smoothness indicator a
# Gram matrix of its derivatives.

def _mono(k, a, b):  # int_a^b x^k dx
    return (b ** (k + 1) - a ** (k + 1)) / (k + 1)


def _moment(powers, kind, cell):
    """The average (kind 0) or the first moment in direction kind - 1 of the
    monomial over the unit cell centred at `cell`."""
    v = 1.0
    for d, (p, c) in enumerate(zip(powers, cell)):
        m = _mono(p, c - 0.5, c + 0.5)
        if kind == d + 1:
            m = _mono(p + 1, c - 0.5, c + 0.5) - c * m
        v *= m
    return v


def _gram(powers, degree):
    """sum over 1 <= |l| <= degree of the integral of D^l p D^l q."""
    dim = len(powers[0])
    orders = [(a,) for a in range(1, degree + 1)] if dim == 1 else \
        [(a, b) for a in range(degree + 1) for b in range(degree + 1 - a) if a + b > 0]
    g = np.zeros((len(powers), len(powers)))
    for l in orders:
        for i, p in enumerate(powers):
            for j, q in enumerate(powers):
                v = 1.0
                for d in range(dim):
                    if p[d] < l[d] or q[d] < l[d]:
                        v = 0.0
                        break
                    v *= math.perm(p[d], l[d]) * math.perm(q[d], l[d]) * _mono(p[d] + q[d] - 2 * l[d], -0.5, 0.5)
                g[i, j] += v
    return g


def _candidate(powers, degree, exact_rows, square_rows, data, targets):
    """(values at the targets, smoothness matrix) as maps of the data, a list of
    (kind, cell): the polynomial meets exact_rows and, where there are more
    coefficients, square_rows in least squares.  A target is a point, or
    ("moment", kind)."""
    rows = lambda which: np.array([[_moment(p, *data[k]) for p in powers] for k in which])  # noqa: E731
    n, m = len(powers), len(exact_rows)
    kkt, rhs = np.zeros((n + m, n + m)), np.zeros((n + m, len(data)))
    e = rows(exact_rows)
    kkt[:n, n:], kkt[n:, :n] = e.T, e
    for r, k in enumerate(exact_rows):
        rhs[n + r, k] = 1.0
    if square_rows:
        a = rows(square_rows)
        kkt[:n, :n] = a.T @ a
        for r, k in enumerate(square_rows):
            rhs[:n, k] = a[r]
    coef = np.linalg.solve(kkt, rhs)[:n] if square_rows else np.linalg.solve(e, rhs[n:])
    at = np.array([[_moment(p, t[1], (0.0,) * len(p)) if t[0] == "moment" else
                    np.prod([np.float64(x) ** k for x, k in zip(t, p)]) for p in powers] for t in targets])
    return at @ coef, coef.T @ _gram(powers, degree) @ coef


def _tables(dim, gauss):
    """The limiter's and the reconstruction's (values, smoothness) tables."""
    dev = lambda pairs: [tuple(torch.tensor(t, device=DEVICE) for t in p) for p in pairs]  # noqa: E731
    line = lambda d: [(k,) for k in range(d + 1)]  # noqa: E731
    d5 = [(0, (-1,)), (0, (0,)), (0, (1,)), (1, (-1,)), (1, (1,))]
    own = [("moment", 1)]
    lim = [_candidate(line(4), 4, [0, 1, 2, 3, 4], [], d5, own),
           _candidate(line(1), 1, [0, 1], [], d5, own), _candidate(line(1), 1, [1, 2], [], d5, own)]
    if dim == 1:
        d6 = [(0, (-1,)), (0, (0,)), (0, (1,)), (1, (-1,)), (1, (0,)), (1, (1,))]
        s = math.sqrt(5.0) / 10.0
        pts = [(-0.5,), (0.5,), (-s,), (s,)]
        rec = [_candidate(line(5), 5, range(6), [], d6, pts),
               _candidate(line(2), 2, [0, 1, 4], [], d6, pts), _candidate(line(2), 2, [1, 2, 4], [], d6, pts)]
        return dev(lim), dev(rec)
    plane = lambda d: [(t - b, b) for t in range(d + 1) for b in range(t + 1)]  # noqa: E731
    cells = [(i, j) for j in (-1, 0, 1) for i in (-1, 0, 1)]
    mom = [1, 3, 4, 5, 7]
    d19 = [(0, c) for c in cells] + [(1, cells[k]) for k in mom] + [(2, cells[k]) for k in mom]
    g, _ = _gauss(gauss)
    pts = [(-0.5, y) for y in g] + [(0.5, y) for y in g] + [(x, -0.5) for x in g] + \
          [(x, 0.5) for x in g] + [(x, y) for y in g for x in g]
    exact_rows = list(range(9)) + [11, 16]
    rec = [_candidate(plane(4), 4, exact_rows, [k for k in range(9, 19) if k not in exact_rows], d19, pts)]
    for st in ((0, 1, 3, 4), (1, 2, 4, 5), (3, 4, 6, 7), (4, 5, 7, 8)):
        rec.append(_candidate(plane(2), 2, list(st) + [11, 16], [], d19, pts))
    return dev(lim), dev(rec)


def _combine(tables, gam, d, points):
    """The nonlinear combination at the first `points` targets: d [F, data, K]."""
    beta = [torch.einsum("fik,ij,fjk->fk", d, b, d) for _, b in tables]
    val = [torch.einsum("pi,fik->fpk", v[:points], d) for v, _ in tables]
    tau = (sum((beta[0] - b).abs() for b in beta[1:]) / (len(beta) - 1)) ** 2
    w = [g * (1.0 + tau / (b + EPS)) for g, b in zip(gam, beta)]
    s = sum(w)
    big = (val[0] - sum(g * v for g, v in zip(gam[1:], val[1:]))) / gam[0]
    out = (w[0] / s)[:, None] * big
    for x, v in zip(w[1:], val[1:]):
        out = out + (x / s)[:, None] * v
    return out


def _flux(U, d):
    """The flux in direction d of [C, ...]: Burgers (C = 1) or Euler."""
    if U.shape[0] == 1:
        return 0.5 * U * U
    rho, E, vel = U[0], U[-1], U[1:-1] / U[0]
    p = (GAS - 1.0) * (E - 0.5 * (U[1:-1] * vel).sum(0))
    vn = vel[d]
    f = [rho * vn] + [U[1 + k] * vn + (p if k == d else 0.0) for k in range(len(vel))] + [vn * (E + p)]
    return torch.stack(f)


def _speed(U, d):
    if U.shape[0] == 1:
        return U[0].abs()
    vel = U[1:-1] / U[0]
    p = (GAS - 1.0) * (U[-1] - 0.5 * (U[1:-1] * vel).sum(0))
    return vel[d].abs() + torch.sqrt(GAS * p / U[0])


def _eigen(U, d):
    """(left, right) eigenvectors [K, C, C] of the Jacobian in direction d."""
    if U.shape[0] == 1:
        one = torch.ones(U.shape[1], 1, 1, device=DEVICE, dtype=U.dtype)
        return one, one
    vel = U[1:-1] / U[0]
    q = 0.5 * (vel * vel).sum(0)
    p = (GAS - 1.0) * (U[-1] - U[0] * q)
    c, h = torch.sqrt(GAS * p / U[0]), (U[-1] + p) / U[0]
    one, zero, vn = torch.ones_like(c), torch.zeros_like(c), vel[d]
    cols = []
    for s in (-1.0, 0.0, 1.0):
        v = [vel[k] + (s * c if k == d else 0.0) for k in range(len(vel))]
        cols.append(torch.stack([one] + v + [h + s * vn * c if s else q]))
    if len(vel) == 2:  # the shear wave
        t = 1 - d
        cols.insert(2, torch.stack([zero] + [one if k == t else zero for k in range(2)] + [vel[t]]))
    R = torch.stack(cols, dim=1).permute(2, 0, 1)  # [K, component, field]
    return torch.linalg.inv(R), R


def _in_fields(tables, gam, U, d, data, points):
    """_combine in the characteristic fields of U [C, K]: data [C, n, K]."""
    L, R = _eigen(U, d)
    ch = _combine(tables, gam, torch.einsum("kfc,cnk->fnk", L, data), points)
    return torch.einsum("kcf,fpk->cpk", R, ch)


class _Exact1D:
    """Instances of sizes n_b, each with three ghost cells a side, in one row."""

    def __init__(self, case):
        self.gam = [0.98, 0.01, 0.01]
        self.lim, self.rec = _tables(1, 0)
        x0, x1, _, _ = _domain(case)
        sizes = _batch_sizes(case)
        src, inst, mirror, off = [], [], [], 0
        for b, n in enumerate(sizes):
            i = np.arange(-3, n + 3)
            ghost = (i < 0) | (i >= n)
            if case["bc"] == "periodic":
                j = i % n
            elif case["bc"] == "outflow":
                j = np.clip(i, 0, n - 1)
            else:
                j = np.where(i < 0, -1 - i, np.where(i >= n, 2 * n - 1 - i, i))
            src.append(j + off)
            mirror.append(ghost & (case["bc"] == "reflective"))
            inst.append(np.full(n + 6, b))
            off += n
        t = lambda a: torch.tensor(np.concatenate(a), device=DEVICE)  # noqa: E731
        self.src, self.inst, mir = t(src), t(inst), t(mirror)
        i = np.concatenate([np.arange(-3, n + 3) for n in sizes])
        n = np.concatenate([np.full(k + 6, k) for k in sizes])
        self.own = torch.tensor((i >= 0) & (i < n), device=DEVICE)
        C = 3 if case["system"] == "euler" else 1
        sign = torch.ones(C, 2, len(i), device=DEVICE, dtype=torch.float64)
        sign[:, 1, mir] = -1.0
        if C == 3:
            sign[1] = -sign[1] * mir + sign[1] * ~mir
        self.sign, self.C = sign, C
        self.dx = torch.tensor([(x1 - x0) / k for k in sizes], device=DEVICE, dtype=torch.float64)
        self.dxc = self.dx[self.inst]
        self.cfl, self.sizes = case["cfl"], sizes

    def alpha(self, U):
        a = torch.zeros(len(self.sizes), device=DEVICE, dtype=torch.float64)
        return a.scatter_reduce(0, self.inst[self.own], _speed(U[:, 0], 0), "amax")

    def operator(self, U):
        """L, the limited state, the flags: U [C, 2, cells]."""
        m, p = (lambda a: torch.roll(a, 1, -1)), (lambda a: torch.roll(a, -1, -1))
        P = U[:, :, self.src] * self.sign
        u, v = P[:, 0], P[:, 1]
        left = (u[1] / u[0] if self.C == 3 else u[0]) >= 0.0
        jump = torch.where(left, (u - 6.0 * v) - m(u + 6.0 * v), (u + 6.0 * v) - p(u - 6.0 * v))
        bad = jump.abs() > 0.5 * self.dxc * u.abs().clamp(min=1e-12)
        flag = bad[0] | bad[2] if self.C == 3 else bad[0]
        flag[0] = flag[-1] = False
        k = flag.nonzero()[:, 0]
        vl = v.clone()
        if len(k):
            data = torch.stack([u[:, k - 1], u[:, k], u[:, k + 1], v[:, k - 1], v[:, k + 1]], dim=1)
            vl[:, k] = _in_fields(self.lim, self.gam, u[:, k], 0, data, 1)[:, 0]
        data = torch.stack([m(u), u, p(u), m(vl), vl, p(vl)], dim=1)
        pts = torch.einsum("pi,cik->cpk", self.rec[0][0], data)
        k = (flag | m(flag) | p(flag)).nonzero()[:, 0]
        if len(k):
            pts[:, :2, k] = _in_fields(self.rec, self.gam, u[:, k], 0, data[:, :, k], 2)
        F = [_flux(pts[:, q], 0) for q in range(4)]
        a = self.alpha(U)[self.inst]
        lo = 0.5 * (m(F[1]) + F[0]) - 0.5 * a * (pts[:, 0] - m(pts[:, 1]))
        hi = 0.5 * (F[1] + p(F[0])) - 0.5 * a * (p(pts[:, 0]) - pts[:, 1])
        vol = (F[0] + F[1]) / 12.0 + (F[2] + F[3]) * (5.0 / 12.0)
        L = torch.stack([-(hi - lo) / self.dxc, (vol - 0.5 * (lo + hi)) / self.dxc], dim=1)
        W = torch.stack([u, vl], dim=1)
        return L[:, :, self.own], W[:, :, self.own], flag[self.own]

    def run(self, U, steps):
        t = torch.zeros_like(self.dx)
        for _ in range(steps):
            dt1 = self.cfl * self.dx / self.alpha(U)
            dt = dt1[self.inst[self.own]]
            L, W0, _ = self.operator(U)
            U = W0 + dt * L
            L, W, _ = self.operator(U)
            U = 0.75 * W0 + 0.25 * (W + dt * L)
            L, W, _ = self.operator(U)
            U = (W0 + 2.0 * (W + dt * L)) / 3.0
            t = t + dt1
        return U, t

    def pack(self, U):
        """[C, 2, cells] -> the instances one after the other."""
        return torch.cat([x.reshape(-1) for x in torch.split(U, self.sizes, dim=-1)])

    def unpack(self, u):
        parts, off = [], 0
        for n in self.sizes:
            parts.append(u[off:off + 2 * self.C * n].reshape(self.C, 2, n))
            off += 2 * self.C * n
        return torch.cat(parts, dim=-1)


class _Exact2D:
    def __init__(self, case):
        self.gam = [0.96, 0.01, 0.01, 0.01, 0.01]
        self.lim, self.rec = _tables(2, case["gauss"])
        self.gauss, self.cfl = case["gauss"], case["cfl"]
        x0, x1, y0, y1 = _domain(case)
        nx, ny = case["nx"], case["ny"]
        self.dx, self.dy = (x1 - x0) / nx, (y1 - y0) / ny

        def ghosts(n):
            i = np.arange(-3, n + 3)
            i = i % n if case["bc"] == "periodic" else np.clip(i, 0, n - 1)
            return torch.tensor(i, device=DEVICE)
        self.ii, self.jj = ghosts(nx), ghosts(ny)

    @staticmethod
    def _near(a, i, j, margin):
        """a at the cells (i, j) away, `margin` fewer cells a side."""
        h, w = a.shape[-2] - 2 * margin, a.shape[-1] - 2 * margin
        return a[..., margin + j:margin + j + h, margin + i:margin + i + w]

    def alphas(self, U):
        return _speed(U[:, 0], 0).max(), _speed(U[:, 0], 1).max()

    def flags(self, U):
        """Of the cells and two ghost cells a side."""
        P = U[:, :, self.jj][:, :, :, self.ii]
        C = P.shape[0]
        near = lambda a, i, j: self._near(a, i, j, 1)  # noqa: E731
        u, v, w = P[:, 0], P[:, 1], P[:, 2]
        c = near(u, 0, 0)
        velx, vely = (c[1] / c[0], c[2] / c[0]) if C == 4 else (c[0], c[0])
        jx = torch.where(velx >= 0.0, near(u - 6 * v, 0, 0) - near(u + 6 * v, -1, 0),
                         near(u + 6 * v, 0, 0) - near(u - 6 * v, 1, 0))
        jy = torch.where(vely >= 0.0, near(u - 6 * w, 0, 0) - near(u + 6 * w, 0, -1),
                         near(u + 6 * w, 0, 0) - near(u - 6 * w, 0, 1))
        h = 0.5 * math.sqrt(self.dx ** 2 + self.dy ** 2)
        bad = (self.dy * jx + self.dx * jy).abs() > h * (self.dx + self.dy) * c.abs().clamp(min=1e-12)
        return bad[0] | bad[3] if C == 4 else bad[0]

    def operator(self, U, flag, ax, ay):
        """L and the limited state: U [C, 3, ny, nx], flag from flags()."""
        P = U[:, :, self.jj][:, :, :, self.ii]
        C, g = P.shape[0], self.gauss
        u = P[:, 0]
        j, i = (x + 1 for x in flag.nonzero(as_tuple=True))
        lim = [P[:, 1], P[:, 2]]
        if len(i):
            for d, (si, sj) in enumerate(((1, 0), (0, 1))):
                mom = lim[d]
                data = torch.stack([u[:, j - sj, i - si], u[:, j, i], u[:, j + sj, i + si],
                                    mom[:, j - sj, i - si], mom[:, j + sj, i + si]], dim=1)
                new = _in_fields(self.lim, self.gam[:3], u[:, j, i], d, data, 1)[:, 0]
                lim[d] = mom.index_put((torch.arange(C, device=DEVICE)[:, None], j[None], i[None]), new)
        cells = [(a, b) for b in (-1, 0, 1) for a in (-1, 0, 1)]
        mom = [cells[k] for k in (1, 3, 4, 5, 7)]
        data = torch.stack([self._near(u, a, b, 2) for a, b in cells] +
                           [self._near(lim[0], a, b, 2) for a, b in mom] +
                           [self._near(lim[1], a, b, 2) for a, b in mom], dim=1)  # one ghost cell a side
        pts = torch.einsum("pi,cihw->cphw", self.rec[0][0], data)
        near = torch.zeros_like(self._near(flag, 0, 0, 1))
        for a, b in cells:
            near = near | self._near(flag, a, b, 1)
        j, i = near.nonzero(as_tuple=True)
        if len(i):
            own = u[:, j + 2, i + 2]
            xf = _in_fields(self.rec, self.gam, own, 0, data[:, :, j, i], 4 * g)[:, :2 * g]
            yf = _in_fields(self.rec, self.gam, own, 1, data[:, :, j, i], 4 * g)[:, 2 * g:]
            at = (torch.arange(C, device=DEVICE)[:, None, None], torch.arange(4 * g, device=DEVICE)[None, :, None],
                  j[None, None], i[None, None])
            pts = pts.index_put(at, torch.cat([xf, yf], dim=1))
        del data
        me = lambda q: self._near(pts[:, q], 0, 0, 1)  # noqa: E731
        to = lambda q, a, b: self._near(pts[:, q], a, b, 1)  # noqa: E731

        def lf(a, b, d, alpha):
            return 0.5 * (_flux(a, d) + _flux(b, d)) - 0.5 * alpha * (b - a)
        x, w = _gauss(g)
        sx = sxs = sxe = sy = sys_ = sye = vx = vy = 0.0
        for k in range(g):
            lo, hi = lf(to(g + k, -1, 0), me(k), 0, ax), lf(me(g + k), to(k, 1, 0), 0, ax)
            bo, up = lf(to(3 * g + k, 0, -1), me(2 * g + k), 1, ay), lf(me(3 * g + k), to(2 * g + k, 0, 1), 1, ay)
            sx, sxs, sxe = sx + w[k] * (hi - lo), sxs + w[k] * (hi + lo), sxe + w[k] * x[k] * (hi - lo)
            sy, sys_, sye = sy + w[k] * (up - bo), sys_ + w[k] * (up + bo), sye + w[k] * x[k] * (up - bo)
            for l in range(g):
                q = me(4 * g + l * g + k)
                vx, vy = vx + w[k] * w[l] * _flux(q, 0), vy + w[k] * w[l] * _flux(q, 1)
        L = torch.stack([-sx / self.dx - sy / self.dy,
                         -0.5 * sxs / self.dx + vx / self.dx - sye / self.dy,
                         -sxe / self.dx - 0.5 * sys_ / self.dy + vy / self.dy], dim=1)
        W = torch.stack([u, lim[0], lim[1]], dim=1)[:, :, 3:-3, 3:-3]
        return L, W

    def switches(self, U):
        return (self.flags(U),) + self.alphas(U)

    def step(self, U, tape=None):
        """One step and what it decided; with a tape, that step with its decisions."""
        got = []

        def op(V, k):
            s = tape[0][k] if tape else self.switches(V)
            got.append(s)
            return self.operator(V, *s)
        dt = tape[1] if tape else self.cfl / (self.alphas(U)[0] / self.dx + self.alphas(U)[1] / self.dy)
        L, W0 = op(U, 0)
        V = W0 + dt * L
        L, W = op(V, 1)
        V = 0.75 * W0 + 0.25 * (W + dt * L)
        L, W = op(V, 2)
        return (W0 + 2.0 * (W + dt * L)) / 3.0, (got, dt)


def exact(case, seed):
    u = _initial(case, seed).to(torch.float64)
    if case["kind"].endswith("1d"):
        s = _Exact1D(case)
        U = s.unpack(u.reshape(-1))
        if case["kind"] == "rhs1d":
            L, W, flags = s.operator(U)
            return {"rhs": L, "ulim": W, "flags": None}
        U, t = s.run(U, case["steps"])
        if case["kind"] == "batch1d":
            return {"state": s.pack(U), "times": t}
        return {"state": U, "t": float(t[0])}
    s = _Exact2D(case)
    if case["kind"] == "rhs2d":
        sw = s.switches(u)
        L, W = s.operator(u, *sw)
        return {"rhs": L, "ulim": W, "flags": None}
    t, seen, tapes = 0.0, [], []
    for _ in range(case["steps"]):
        with torch.no_grad():
            new, tape = s.step(u)
        if case["kind"] == "adjoint2d":
            seen.append(u)
            tapes.append(tape)
        u, t = new, t + float(tape[1])
    if case["kind"] == "run2d":
        return {"state": u, "t": t}
    grad = torch.zeros_like(u)
    grad[0, 0] = 2.0 * u[0, 0]
    for v, tape in zip(reversed(seen), reversed(tapes)):
        v = v.detach().requires_grad_(True)
        out, _ = s.step(v, tape)
        grad, = torch.autograd.grad(out, v, grad)
    return {"state": u, "grad": grad}
