"""The work that users of this package have it do, as cases that can be timed.

A case is one pass through the public entry points on data that is already on the GPU, with a plan that
the program keeps: a solve in one of the three arithmetic modes, a refined solve, a solve with face data,
a solve with its gradient, or a batch of solves.  ``listed`` holds the workloads of this repository's
benchmark and configurations; ``draw`` gives others of the same kinds, with any sizes the solver takes.
"""
import math

import torch

import paper_1909_05423_gb300 as pp
from paper_1909_05423_gb300 import workloads

# Largest number of grid points that draw() gives: half of the largest listed grid, so that no drawn
# case (run-time line lengths, refined solves, forward and adjoint) costs more than that one.
DRAW_POINTS = 2 ** 28


def listed():
    cube = lambda n: {"nx": n, "ny": n, "nz": n}  # noqa: E731
    return [
        # The smallest call: a manufactured source on a small cube with fixed walls, as in a convergence
        # study or inside a time step of a small simulation.  Latency and launches count.
        {"name": "modes_32_f64", "kind": "solve", **cube(32), "bc": "DDDDDD", "dtype": "f64", "source": "modes"},
        # A middle-sized simulation grid with mixed walls, near the size of the L2 cache.
        {"name": "cube_256_f64", "kind": "solve", **cube(256), "bc": "NNDDNN", "dtype": "f64", "source": "uniform"},
        # The headline: the largest cube, double precision, tuned plan.
        {"name": "cube_1024_f64", "kind": "solve", **cube(1024), "bc": "NNDDNN", "dtype": "f64", "source": "uniform",
         "autotune": True},
        # The same grid where single-precision transforms are enough.
        {"name": "cube_1024_mixed", "kind": "solve", **cube(1024), "bc": "NNDDNN", "dtype": "mixed_f64io",
         "source": "uniform", "autotune": True},
        # Periodic turbulence boxes: complex lines along y and cyclic systems along z.
        {"name": "periodic_512_f64", "kind": "solve", **cube(512), "bc": "PPPPPP", "dtype": "f64", "source": "modes"},
        # Single-precision transforms with one refinement step: most of the digits at less cost.
        {"name": "refined_512", "kind": "refined", **cube(512), "bc": "NNNNNN", "dtype": "mixed_f64io",
         "source": "modes"},
        # Many small uneven grids at once (subdomains, parameter studies), in both I/O types.
        {"name": "batch_64_f64", "kind": "batch", "count": 64, "grids": 5, "dtype": "f64", "source": "uniform"},
        {"name": "batch_64_f32", "kind": "batch", "count": 64, "grids": 5, "dtype": "mixed_f32io", "source": "uniform"},
        # Fitting a source to a target field: the solve and its gradient.
        {"name": "adjoint_256_f64", "kind": "adjoint", **cube(256), "bc": "NNDDNN", "dtype": "f64", "source": "blobs"},
        # Few modes on long lines: channels, columns, and the shapes on which tridiagonal solvers are compared.
        {"name": "long_lines_4095", "kind": "solve", "nx": 64, "ny": 64, "nz": 4095, "bc": "PPPPDD", "dtype": "f64",
         "source": "uniform"},
        # Sizes that suit the geometry and not the machine: factors 5 and 7, an odd number of planes, and
        # another condition on every face.
        {"name": "ragged_140_f64", "kind": "solve", "nx": 120, "ny": 140, "nz": 99, "bc": "DNPPND", "dtype": "f64",
         "source": "uniform"},
        # Prescribed values and fluxes on the faces, single-precision data.
        {"name": "faces_384_f32", "kind": "faces", "nx": 384, "ny": 192, "nz": 300, "bc": "DNNDDD",
         "dtype": "mixed_f32io", "source": "uniform"},
    ]


def _smooth(limit):
    """Even 2^a 3^b 5^c 7^d up to limit: the lengths that x and y take."""
    out = []
    for n in range(2, limit + 1, 2):
        m = n
        for q in (2, 3, 5, 7):
            while m % q == 0:
                m //= q
        if m == 1:
            out.append(n)
    return out


def _draw_bc(rng):
    return "".join("PP" if rng.random() < 1 / 3 else rng.choice("ND") + rng.choice("ND") for _ in range(3))


def _draw_side(rng, centre):
    """A length near `centre` (within a factor of about 2): half of them 2^a or 3 2^a, the others any the
    solver takes."""
    want = centre * 2.0 ** rng.uniform(-1, 1)
    plain = [n for a in range(4, 12) for n in (2 ** a, 3 * 2 ** (a - 1)) if n <= 2048]
    pool = plain if rng.random() < 0.5 else [n for n in _smooth(2048) if n >= 12]
    return min(pool, key=lambda n: abs(math.log(n / want)) + 1e-3 * rng.random())


def draw(rng):
    dtype = rng.choice(["f64", "f64", "f64", "mixed_f64io", "mixed_f32io"])
    kind = rng.choices(["solve", "refined", "faces", "adjoint", "batch"], [6, 1, 1, 1, 1])[0]
    source = rng.choice(["uniform", "uniform", "modes", "blobs"])
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(4, 48), "grids": rng.randrange(1 << 20),
                "dtype": rng.choice(["f64", "mixed_f32io"]), "source": source}
    if kind == "refined":
        dtype = "mixed_f64io"
    points = 2.0 ** rng.uniform(15, math.log2(DRAW_POINTS))
    while True:
        if rng.random() < 0.2:  # few modes on long lines
            nx, ny = _draw_side(rng, 64), _draw_side(rng, 64)
            nz = int(2.0 ** rng.uniform(7, 12))
        else:
            side = points ** (1 / 3)
            nx, ny = _draw_side(rng, side), _draw_side(rng, side)
            nz = max(5, round(points / (nx * ny)))
        if 2 ** 14 <= nx * ny * nz <= DRAW_POINTS and nz <= 4096:
            break
    case = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "bc": _draw_bc(rng), "dtype": dtype, "source": source}
    if kind == "solve" and rng.random() < 0.25:
        case["autotune"] = True
    return case


def _grids(case):
    """(shape, boundary conditions) of every grid of a case."""
    if case["kind"] == "batch":
        return workloads.batched_grids(case["grids"], count=case["count"])
    return [((case["nz"], case["ny"], case["nx"]), case["bc"])]


def _spacing(shape):
    """The unit cube in x, and cells of the same size in y and z."""
    h = 1.0 / shape[2]
    return (h, h, h)


def _io(case):
    return torch.float32 if case["dtype"] == "mixed_f32io" else torch.float64


def _centres(n, device):
    return (torch.arange(n, dtype=torch.float64, device=device) + 0.5) / n


def _source(case, shape, gen, device):
    """A source of a grid, in FP64: noise, a few smooth products of cosines and sines, or Gaussian blobs."""
    nz, ny, nx = shape
    if case["source"] == "uniform":
        f = torch.rand(shape, dtype=torch.float64, device=device, generator=gen).mul_(2.0).sub_(1.0)
        return f.sub_(f.mean())
    z, y, x = (_centres(n, device) for n in shape)
    f = torch.zeros(shape, dtype=torch.float64, device=device)
    par = torch.rand((8, 10), dtype=torch.float64, device=device, generator=gen).cpu()
    for p in par[:4] if case["source"] == "modes" else par:
        if case["source"] == "modes":
            g = [torch.cos(2.0 * math.pi * (int(8 * p[a]) + 1) * c + 2.0 * math.pi * p[3 + a])
                 for a, c in enumerate((z, y, x))]
        else:
            w = 0.03 + 0.07 * float(p[6])
            g = [torch.exp(-((c - 0.2 - 0.6 * float(p[a])) ** 2) / (2.0 * w * w)) for a, c in enumerate((z, y, x))]
        t = g[0][:, None, None] * g[1][None, :, None]
        f.addcmul_(t.mul_(2.0 * float(p[7]) - 1.0), g[2][None, None, :])
    return f


def _inputs(case, seed, device):
    """What the solver is given: the sources of all grids, face data and a target field where the case has them."""
    gen = torch.Generator(device=device)
    gen.manual_seed(seed)
    dt = _io(case)
    fs = [_source(case, shape, gen, device).to(dt) for shape, _ in _grids(case)]
    shape, bc = _grids(case)[0]
    nz, ny, nx = shape
    faces = target = None
    if case["kind"] == "faces":
        shapes = [(nz, ny), (nz, ny), (nz, nx), (nz, nx), (ny, nx), (ny, nx)]
        faces = [None if b == "P" else torch.rand(s, dtype=torch.float64, device=device, generator=gen).to(dt)
                 for b, s in zip(bc, shapes)]
    if case["kind"] == "adjoint":
        target = torch.rand(shape, dtype=torch.float64, device=device, generator=gen).sub_(0.5).mul_(1e-3).to(dt)
    return fs, faces, target


def prepare(case, seed):
    fs, faces, target = _inputs(case, seed, "cuda")
    options = {"autotune": 1} if case.get("autotune") else None
    plans = [pp.Plan(shape, bc, _spacing(shape), case["dtype"], options) for shape, bc in _grids(case)]
    if case["kind"] == "adjoint":
        fs[0].requires_grad_(True)
    return {"kind": case["kind"], "plans": plans, "fs": fs, "faces": faces, "target": target,
            "us": [torch.empty_like(f, requires_grad=False) for f in fs]}


def run(state):
    kind, plan, f, u = state["kind"], state["plans"][0], state["fs"][0], state["us"][0]
    if kind == "batch":
        return pp.solve_batched(state["plans"], state["fs"], state["us"])
    if kind == "refined":
        return plan.solve_refined(f, out=u)
    if kind == "faces":
        return plan.solve_bc(f, state["faces"], out=u)
    if kind == "adjoint":
        # the gradient of |S f - target|^2 / 2
        u = pp.PoissonSolve.apply(f, plan)
        (g,) = torch.autograd.grad(u, f, u.detach() - state["target"])
        return [u.detach(), g]
    return plan.solve(f, out=u)


def work(case):
    """The sources (and face data, target) read once and the solutions (and gradient) written once; the
    real line transforms at 2.5 N log2 N operations, forward and back in x and y, and 8 operations a
    point along z."""
    e = 4 if case["dtype"] == "mixed_f32io" else 8
    total = flops = 0
    for (nz, ny, nx), _ in _grids(case):
        n = nx * ny * nz
        total += 2 * e * n
        flops += n * (5.0 * math.log2(nx) + 5.0 * math.log2(ny) + 8.0)
    if case["kind"] == "faces":
        total += 2 * e * (nz * ny + nz * nx + ny * nx)
    if case["kind"] == "adjoint":
        total, flops = total + 2 * e * n, 2 * flops
    if case["kind"] == "refined":
        flops = 2 * flops + 16.0 * n
    return {"bytes": total, "flops": flops}


def _eigen(lo, hi, n, h, device):
    """Eigenvalues and orthonormal eigenvectors (rows) of the second difference along one axis.  Angles are
    reduced in integers, and the eigenvalues are -4 sin^2 / h^2, so nothing cancels."""
    k = torch.arange(n, device=device)[:, None]
    j = torch.arange(n, device=device)[None, :]

    def trig(fn, num, den):  # fn(pi num / den)
        return fn((num % (2 * den)).double() * (math.pi / den))

    if lo == "P":
        half = (k + 1) // 2  # 0, 1, 1, 2, 2, ...: constant, cos, sin, cos, sin, ...
        v = torch.where(k % 2 == 1, trig(torch.cos, 2 * half * j, n), trig(torch.sin, 2 * half * j, n))
        v[0] = 1.0
        theta = half[:, 0].double() * (math.pi / n)
    else:
        if lo == hi:
            num, den = ((k, 2 * n) if lo == "N" else (k + 1, 2 * n))
        else:
            num, den = 2 * k + 1, 4 * n
        v = trig(torch.cos if lo == "N" else torch.sin, num * (2 * j + 1), den)
        theta = num[:, 0].double() * (math.pi / den)
    v = v / torch.linalg.vector_norm(v, dim=1, keepdim=True)
    return -4.0 * torch.sin(theta) ** 2 / (h * h), v


def _solve64(f, bc, spacing):
    """The discrete solution by dense eigenvector products along every axis, in FP64 (zero mean where the
    operator is singular)."""
    h = dict(zip((2, 1, 0), spacing))
    lam, vec = zip(*(_eigen(bc[2 * (2 - a)], bc[2 * (2 - a) + 1], f.shape[a], h[a], f.device) for a in range(3)))
    nz, ny, nx = f.shape
    t = (f.reshape(-1, nx) @ vec[2].T).reshape(f.shape)
    t = torch.matmul(vec[1], t)
    t = (vec[0] @ t.reshape(nz, -1)).reshape(f.shape)
    for k in range(nz):
        s = lam[0][k] + lam[1][:, None] + lam[2][None, :]
        t[k] = torch.where(s == 0, 0.0, t[k] / s)
    t = (vec[0].T @ t.reshape(nz, -1)).reshape(f.shape)
    t = torch.matmul(vec[1].T.contiguous(), t)
    return (t.reshape(-1, nx) @ vec[2]).reshape(f.shape)


def _folded(f, faces, bc, spacing):
    """The source with the face data's ghost terms: 2 g / h^2 next to a Dirichlet face, q / h next to a
    Neumann face."""
    f = f.clone()
    for i, g in enumerate(faces):
        if g is not None:
            axis, h = 2 - i // 2, spacing[i // 2]
            f.select(axis, -1 if i % 2 else 0).sub_(g.double() * (2.0 / (h * h) if bc[i] == "D" else 1.0 / h))
    return f


def exact(case, seed, device="cuda"):
    fs, faces, target = _inputs(case, seed, device)
    out = []
    for (shape, bc), f in zip(_grids(case), fs):
        f = f.double()
        if faces is not None:
            f = _folded(f, faces, bc, _spacing(shape))
        u = _solve64(f, bc, _spacing(shape))
        out.append(u)
    if case["kind"] == "adjoint":
        return [u, _solve64(u - target.double(), bc, _spacing(shape))]
    return out if case["kind"] == "batch" else u
