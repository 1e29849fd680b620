"""The work that users of the implicit reaction-diffusion solver have it do, as timed cases.

A case is one call (or one served batch) through the Python binding: an implicit time step of a
`Solver`, an application of the preconditioner, or a mix of requests through `Batch`.  Problems are
the repository's own workloads (workloads.py) on grids from 64 x 64 to 8192 x 8192; their physical
parameters are taken from there and the initial states follow the same recipes, drawn on the GPU.
"""
import math

import numpy as np
import torch

from paper_2305_03945_gb300 import rd, workloads as WL

# One entry per equation: the workload whose parameters it takes, and the initial state's recipe.
_PHYSICS = {
    "ac_periodic": lambda: WL.config_allen_cahn_periodic(64).problem.replace(tol=1e-11, tol_kind="f_rel"),
    "ac_neumann": lambda: WL.config_allen_cahn_neumann(64).problem,
    "ch_split": lambda: WL.config_cahn_hilliard_split(64).problem,
    # the implicit Cahn-Hilliard equation of the seven-circle example with the split example's scales
    "ch_implicit": lambda: WL.config_cahn_hilliard_split(64).problem.replace(kind="ch_implicit"),
    "gray_scott": lambda: WL.config_gray_scott(64).problem,
    "schnakenberg": lambda: WL.config_schnakenberg(64).problem.replace(tol=1e-11, tol_kind="f_rel"),
    "fch": lambda: WL.config_fch(64).problem,
}
# PDHG iterations one step takes (FP64), measured on the workloads above: the operation count of a
# step is this many iterations.
_ITERS = {"ac_periodic": 27, "ac_neumann": 14, "ch_split": 7, "ch_implicit": 21, "gray_scott": 45,
          "schnakenberg": 20, "fch": 280}


def _case(do, eq, nx, ny, nz=1, bc="periodic", precision="fp32_dc", autotune=0, dt=1.0, **more):
    return dict(do=do, eq=eq, nx=nx, ny=ny, nz=nz, bc=bc, precision=precision, autotune=autotune, dt=dt, **more)


def listed():
    return [
        # the operator call alone, as a user's own iteration calls it: smallest launches, FP64, two
        # species, Neumann
        dict(_case("precond", "schnakenberg", 128, 128, bc="neumann", precision="fp64"), name="precond_128x2_fp64"),
        # the paper's small Allen-Cahn example: one step, latency-bound
        dict(_case("step", "ac_periodic", 64, 64), name="ac_periodic_64_dc"),
        # the paper's two-species example in the default precision (plain FP64)
        dict(_case("step", "schnakenberg", 128, 128, bc="neumann", precision="fp64"), name="schnakenberg_128_fp64"),
        # the paper's sixth-order example, built in FP64 only
        dict(_case("step", "fch", 128, 128, precision="fp64"), name="fch_128_fp64"),
        # an elongated grid with the fully implicit equation and Neumann walls, default options
        dict(_case("step", "ch_implicit", 1024, 128, bc="neumann"), name="ch_implicit_1024x128_dc"),
        # the benchmark's 2-D workloads with its options (tiles measured when the solver is made)
        dict(_case("step", "ch_split", 512, 512, autotune=1), name="ch_split_512_dc"),
        dict(_case("step", "ac_neumann", 1024, 1024, bc="neumann", autotune=1), name="ac_neumann_1024_dc"),
        dict(_case("step", "gray_scott", 2048, 2048, autotune=1), name="gray_scott_2048_dc"),
        # the same Allen-Cahn step in the default precision (plain FP64) and default options
        dict(_case("step", "ac_neumann", 1024, 1024, bc="neumann", precision="fp64"), name="ac_neumann_1024_fp64"),
        # the serving mix's cube as a single solve
        dict(_case("step", "ac_periodic", 128, 128, 128), name="ac_periodic_128x3_dc"),
        # the largest grid: lines of 8192 points
        dict(_case("step", "ac_periodic", 8192, 8192), name="ac_periodic_8192_dc"),
        # serving: eight requests of uneven sizes, kinds and boundaries submitted together
        dict(_case("batch", "mix", 512, 512, requests=8, mix=1), name="serving_mix_8"),
    ]


def _pick(rng, lo, hi):
    return 1 << rng.randint(lo, hi)


def draw(rng):
    """Sides are powers of two (the library takes no others), each axis on its own; the time step is
    spread over a factor of four below the workload's."""
    dt = round(math.exp(rng.uniform(math.log(0.25), 0.0)), 4)
    family = rng.choice(("dc", "dc", "dc", "fp64", "cube", "precond", "long", "batch"))
    bc = rng.choice(("periodic", "neumann"))
    if family == "dc":
        eq = rng.choice(("ac_periodic", "ac_neumann", "ch_split", "ch_implicit", "gray_scott", "schnakenberg"))
        return _case("step", eq, _pick(rng, 6, 11), _pick(rng, 6, 11), bc=bc, autotune=rng.randint(0, 1), dt=dt)
    if family == "fp64":
        eq = rng.choice(("ac_periodic", "ac_neumann", "ch_split", "gray_scott", "schnakenberg"))
        return _case("step", eq, _pick(rng, 6, 10), _pick(rng, 6, 10), bc=bc, precision="fp64", dt=dt)
    if family == "cube":
        eq = rng.choice(("ac_periodic", "ch_split"))
        return _case("step", eq, _pick(rng, 5, 7), _pick(rng, 5, 7), _pick(rng, 5, 7), bc=bc, dt=dt)
    if family == "precond":
        eq = rng.choice(("ac_periodic", "ch_split", "schnakenberg"))
        return _case("precond", eq, _pick(rng, 6, 11), _pick(rng, 6, 11), bc=bc, precision="fp64", dt=dt)
    if family == "long":
        sides = [_pick(rng, 8, 12), _pick(rng, 12, 13)]
        rng.shuffle(sides)
        return _case("step", "ac_periodic", sides[0], sides[1], bc=bc, dt=dt)
    return _case("batch", "mix", 512, 512, requests=rng.randint(2, 10), mix=rng.randint(2, 1 << 20), dt=dt)


# ---------------------------------------------------------------------------------------------
# problems and initial states
# ---------------------------------------------------------------------------------------------

def _problem(case):
    pb = _PHYSICS[case["eq"]]()
    pb = pb.replace(nx=case["nx"], ny=case["ny"], nz=case["nz"], bc=case["bc"], dt=pb.dt * case["dt"], lz=pb.lx)
    # an elongated grid keeps the workload's mesh width along its shorter axes as a user's would:
    # the domain grows with the side, the cells stay square
    n = min(case["nx"], case["ny"]) if case["nz"] == 1 else min(case["nx"], case["ny"], case["nz"])
    return pb.replace(lx=pb.lx * case["nx"] / n, ly=pb.ly * case["ny"] / n, lz=pb.lx * case["nz"] / n)


def _uniform(g, shape, lo, hi):
    return torch.rand(shape, dtype=torch.float64, device="cuda", generator=g) * (hi - lo) + lo


def _initial(case, pb, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    eq, shape = case["eq"], pb.shape
    if case["do"] == "precond":  # a residual field: rough, every mode present
        return torch.randn(shape, dtype=torch.float64, device="cuda", generator=g)
    if eq == "ac_periodic":
        return _uniform(g, shape, -0.05, 0.05)
    if eq == "ac_neumann":  # tanh of smoothed noise, 8 cells wide
        x = torch.randn(shape, dtype=torch.float64, device="cuda", generator=g)
        for axis in (-1, -2):
            n = shape[axis]
            k = torch.arange(n, dtype=torch.float64, device="cuda")
            k = torch.minimum(k, n - k) * (2 * math.pi / n)
            k = torch.exp(-0.5 * (8.0 * k) ** 2)
            k = k if axis == -1 else k[:, None]
            x = torch.fft.ifft(torch.fft.fft(x, dim=axis) * k, dim=axis).real
        return torch.tanh(x / x.std()).contiguous()
    if eq in ("ch_split", "ch_implicit"):
        u = _uniform(g, shape, -0.1, 0.1)
        return u - u.mean()
    if eq == "gray_scott":  # ten patches of (1/2, 1/4) in (1, 0), with 1% noise
        ny, nx = shape[-2:]
        u = torch.zeros(shape, dtype=torch.float64, device="cuda")
        u[0] = 1.0
        at = torch.rand((10, 2), generator=g, dtype=torch.float64, device="cuda").tolist()
        side = max(2, int(min(nx, ny) / 12.8))
        for a, b in at:
            i = (torch.arange(side, device="cuda") + int(a * ny)) % ny
            j = (torch.arange(side, device="cuda") + int(b * nx)) % nx
            u[0, i[:, None], j[None, :]] = 0.5
            u[1, i[:, None], j[None, :]] = 0.25
        return u * (1.0 + _uniform(g, shape, -0.01, 0.01))
    if eq == "schnakenberg":  # the perturbed equilibrium, at a place of its own
        ny, nx = shape[-2:]
        a, b = torch.rand(2, generator=g, dtype=torch.float64, device="cuda").tolist()
        X = ((torch.arange(nx, dtype=torch.float64, device="cuda") + 0.5) / nx)[None, :]
        Y = ((torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5) / ny)[:, None]
        a_s, b_s = pb.p[3], pb.p[4]
        u = a_s + b_s + 1e-3 * torch.exp(-100 * ((X - a) ** 2 + (Y - b) ** 2))
        return torch.stack([u, torch.full_like(u, b_s / (a_s + b_s) ** 2)])
    # sixth order: the paper's initial data, shifted
    ny, nx = shape[-2:]
    a, b = (_uniform(g, (2,), 0.0, 2 * math.pi)).tolist()
    X = (torch.arange(nx, dtype=torch.float64, device="cuda") * (2 * math.pi / nx) + a)[None, :]
    Y = (torch.arange(ny, dtype=torch.float64, device="cuda") * (2 * math.pi / ny) + b)[:, None]
    s = torch.sin(X) + torch.sin(Y)
    return (2 * torch.exp(s - 2) + 2.2 * torch.exp(-s - 2) - 1)[None].contiguous()


def _requests(case, seed):
    """The mix: its sizes, kinds, boundaries and step counts belong to the case, its initial states
    to the seed.  The serving mix's grids up to 512 x 512 and a 64-cube, 1 to 3 steps each, every
    step solved as closely as the single solves."""
    r = np.random.Generator(np.random.PCG64(case["mix"]))
    grids = [(64, 64), (128, 128), (256, 256), (512, 512), (256, 128), (64, 64, 64)]
    out = []
    for k in range(case["requests"]):
        grid = grids[k % len(grids)] if case["mix"] == 1 else grids[int(r.integers(len(grids)))]
        eq = ("ac_periodic", "ch_split")[int(r.integers(2))]
        bc = ("periodic", "neumann")[int(r.integers(2))]
        steps = int(r.integers(1, 4))
        nx, ny, nz = grid if len(grid) == 3 else (*grid, 1)
        pb = _problem(_case("step", eq, nx, ny, nz, bc=bc, dt=case["dt"]))
        u = np.random.Generator(np.random.PCG64(1000 * seed + k))
        w = 0.05 if eq == "ac_periodic" else 0.1
        u0 = u.uniform(-w, w, size=pb.shape)
        out.append((eq, pb, u0 if eq == "ac_periodic" else u0 - u0.mean(), steps))
    return out


# ---------------------------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------------------------

def prepare(case, seed):
    if case["do"] == "batch":
        return {"case": case, "batch": rd.Batch(1 << 30, 16), "requests": _requests(case, seed)}
    pb = _problem(case)
    u = _initial(case, pb, seed)
    return {"case": case, "u": u, "out": torch.empty_like(u),
            "solver": rd.Solver(pb, precision=case["precision"], autotune=case["autotune"])}


def run(state):
    case = state["case"]
    if case["do"] == "batch":
        b = state["batch"]
        outs = [b.submit(pb, u0, steps, tag=k)[1] for k, (_, pb, u0, steps) in enumerate(state["requests"])]
        left = len(outs)
        while left > 0:
            done = b.poll(timeout=10.0)
            if not done or any(d["status"] != 0 for d in done):
                raise RuntimeError("a served request failed: %r" % (done,))
            left -= len(done)
        return outs
    if case["do"] == "precond":
        state["solver"].apply_precond(state["u"], state["out"])
    else:
        state["solver"].step(state["u"], state["out"])
    return state["out"]


def work(case):
    """Input and output states once; the operations of the step's iterations: four one-dimensional
    transforms per axis pair (2.5 log2 n per point each way and axis for real data) and the stencils,
    reaction terms and updates (about 40 per point)."""
    if case["do"] == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for eq, pb, u0, steps in _requests(case, 0):
            w = work(_case("step", eq, pb.nx, pb.ny, pb.nz))
            total = {k: total[k] + w[k] * (1 if k == "bytes" else steps) for k in total}
        return total
    comps = 2 if case["eq"] in ("gray_scott", "schnakenberg") else 1
    n = comps * case["nx"] * case["ny"] * case["nz"]
    spectral = 5.0 * math.log2(case["nx"] * case["ny"] * case["nz"])
    if case["do"] == "precond":
        return {"bytes": 16.0 * n, "flops": n * spectral}
    return {"bytes": 16.0 * n, "flops": _ITERS[case["eq"]] * n * (spectral + 40.0)}


# ---------------------------------------------------------------------------------------------
# the same in 64 bits, by torch
# ---------------------------------------------------------------------------------------------

def _solve64(eq, pb, u0, steps, do="step"):
    """`steps` implicit steps from u0 (or one preconditioner solve) on the grid, Neumann walls by even
    reflection into a periodic grid of twice the side: each step is the root of F, found by the
    fixed point U <- U - w A^{-1} F(U) with the constant-coefficient part A of F."""
    axes = [-1, -2] + ([-3] if pb.nz > 1 else [])
    n = {-1: pb.nx, -2: pb.ny, -3: pb.nz}
    h = {-1: pb.lx / pb.nx, -2: pb.ly / pb.ny, -3: pb.lz / pb.nz}
    u = u0
    if pb.bc == "neumann":
        for a in axes:
            u = torch.cat([u, u.flip(a)], dim=a)
    dev = u.device
    mu = torch.zeros((), dtype=torch.float64, device=dev)
    for a in axes:
        m = u.shape[a]
        k = torch.arange(m // 2 + 1 if a == -1 else m, dtype=torch.float64, device=dev)
        v = (4.0 / h[a] ** 2) * torch.sin(math.pi * k / m) ** 2
        mu = mu + v.reshape([-1] + [1] * (-1 - a))

    def lap(x):
        out = None
        for a in axes:
            t = (torch.roll(x, 1, a) + torch.roll(x, -1, a) - 2 * x) / h[a] ** 2
            out = t if out is None else out + t
        return out

    def spectral(x, g):  # x / g in the Fourier basis, g a function of the Laplacian's eigenvalues
        dims = list(reversed(axes))
        return torch.fft.irfftn(torch.fft.rfftn(x, dim=dims) / g, s=[x.shape[d] for d in dims], dim=dims)

    a_, b_, dt, p = pb.a, pb.b, pb.dt, pb.p
    if pb.op == "laplacian":
        D = [a_] if pb.ncomp == 1 else [p[0], p[1]]
        A = [1 + dt * Dc * mu for Dc in D]
    elif pb.op == "functionalized":
        A = [1 + dt * a_ * (2 * b_ - a_) * mu ** 2 + dt * a_ ** 2 * mu ** 3]
    else:
        A = [1 + dt * a_ * mu ** 2]

    def back(x):
        for a in axes:
            x = x.narrow(a, 0, n[a])
        return x.contiguous()

    if do == "precond":
        return back(torch.cat([spectral(u[c:c + 1], A[c] ** 2) for c in range(pb.ncomp)]))

    def F(U, uk):
        if eq in ("ac_periodic", "ac_neumann"):
            return U - uk - dt * (a_ * lap(U) - b_ * (U ** 3 - U))
        if eq == "ch_split":
            return U - uk - dt * lap(-a_ * lap(U) + b_ * (U ** 3 - uk))
        if eq == "ch_implicit":
            return U - uk - dt * lap(-a_ * lap(U) + b_ * (U ** 3 - U))
        if eq == "gray_scott":
            x, y = U[0:1], U[1:2]
            r = x * y * y
            return torch.cat([x - uk[0:1] - dt * (p[0] * lap(x) - r + p[2] * (1 - x)),
                              y - uk[1:2] - dt * (p[1] * lap(y) + r - (p[2] + p[3]) * y)])
        if eq == "schnakenberg":
            x, y = U[0:1], U[1:2]
            r = x * x * y
            return torch.cat([x - uk[0:1] - dt * (p[0] * lap(x) + p[2] * (p[3] - x + r)),
                              y - uk[1:2] - dt * (p[1] * lap(y) + p[2] * (p[4] - r))])
        m = a_ * lap(U) - b_ * (U ** 3 - U)
        return U - uk - dt * lap(a_ * lap(m) - b_ * (3 * U ** 2 - 1) * m + a_ * m)

    w = 0.5 if eq == "fch" else 1.0
    for _ in range(steps):
        uk, U, best, worse = u, u, math.inf, 0
        for it in range(4000):
            f = F(U, uk)
            r = float(f.norm() / uk.norm())
            if not math.isfinite(r):
                return None
            worse = worse + 1 if r > 0.9 * best and w == 1.0 or r >= best else 0
            best = min(best, r)
            if r < 1e-15 or worse >= 4:
                break
            U = U - w * torch.cat([spectral(f[c:c + 1], A[c]) for c in range(pb.ncomp)])
        if best > 1e-10:
            return None
        u = U
    return back(u)


def exact(case, seed):
    if case["do"] == "batch":
        return [_solve64(eq, pb, torch.from_numpy(u0).cuda(), steps) for eq, pb, u0, steps in _requests(case, seed)]
    pb = _problem(case)
    return _solve64(case["eq"], pb, _initial(case, pb, seed), 1, case["do"])
