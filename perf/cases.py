"""What a program has this solver do, as cases that can be timed and checked.

A case is a dict of plain values.  ``kind`` says which calls it stands for:

* ``solve``    one potential of one density: ``set_density``, ``solve``, ``potential`` on a prepared
               ``Grid`` (or ``Grid2D``), the density and the potential on the device or in pinned
               host memory, multigrid or (``levels`` = 1) the single-level solver;
* ``batch``    the same for many grids of uneven sizes through ``solve_batch``;
* ``adjoint``  the differentiable solve: the potential and dL/drho through ``torch.autograd``;
* ``gravity``  the fourth-order acceleration of a potential.

Sizes and options come from this repository's tests, benchmark and workloads.  ``nx``, ``ny``, ``nz``
are cells per axis (``nz`` = 0: a two-dimensional grid), ``bc`` one letter per axis (``d``: Dirichlet,
``p``: periodic), ``box`` the extents, ``density`` the kind of source (``sphere``: a uniform sphere with
the faces of its analytic potential, ``noisy``: the same with 10% noise, ``blobs``: one to four Gaussian
blobs with monopole faces, ``grf``: a Gaussian random field with P(k) ~ k^-3), ``options`` a name in
``OPTIONS``.
"""

import math
import random

import numpy as np
import torch

import paper_2306_05332_gb300 as sg

# The smoother settings that the benchmark's solve, the library's defaults and the paper's own
# Gauss-Seidel smoother take (the defaults with N_pre = 2, N_post = 1 in both of the latter).
OPTIONS = {
    "default": {},
    "bench": dict(rkl_order=2, s_smooth=3, tau_frac=0.9, n_pre=5, n_post=3, inner_n_pre=3, inner_n_post=2),
    "rkl1": dict(rkl_order=1, s_smooth=2, tau_frac=0.75),
    "gsrb": dict(smoother="gsrb"),
}

# Typical V-cycles to a relative residual of 1e-8 (used by work() only).
CYCLES = {"default": 15, "bench": 6, "rkl1": 8, "gsrb": 7}


def listed():
    cube = dict(bc="ddd", box="1,1,1", precision="mixed", options="default", levels=0, tol=1e-8, where="device")
    return [
        # the potential of a small box, as a hydrodynamics step or an optimiser's loop asks for it again
        # and again: launches and round trips count
        dict(cube, name="solve_32", kind="solve", nx=32, ny=32, nz=32, density="blobs"),
        # an ordinary ragged box, periodic along one axis, with cells of three different widths
        dict(cube, name="solve_ragged", kind="solve", nx=112, ny=80, nz=144, density="blobs", bc="pdd",
             box="1.3,1,1.7"),
        # an ordinary cube whose density and potential live in pinned host memory
        dict(cube, name="solve_host_128", kind="solve", nx=128, ny=128, nz=128, density="blobs", where="host"),
        # the benchmark's solve: the uniform sphere at 256^3, five levels
        dict(cube, name="solve_sphere_256", kind="solve", nx=256, ny=256, nz=256, density="sphere",
             options="bench", levels=5, box="2,2,2"),
        # the largest: the periodic Gaussian random field at 512^3
        dict(cube, name="solve_grf_512", kind="solve", nx=512, ny=512, nz=512, density="grf", bc="ppp",
             options="bench", levels=6),
        # double precision throughout, on the sphere, to the tighter tolerance that such a user asks for
        dict(cube, name="solve_fp64_256", kind="solve", nx=256, ny=256, nz=256, density="sphere",
             precision="fp64", options="bench", levels=5, box="2,2,2", tol=1e-10),
        # the paper's own smoother
        dict(cube, name="solve_gsrb_192", kind="solve", nx=192, ny=192, nz=192, density="blobs", options="gsrb"),
        # a two-dimensional problem
        dict(cube, name="solve_2d_1024", kind="solve", nx=1024, ny=1024, nz=0, density="blobs", bc="dd",
             box="1,1"),
        # the single-level accelerated solver on odd extents, in double precision
        dict(cube, name="relax_odd", kind="solve", nx=33, ny=29, nz=37, density="blobs", precision="fp64",
             levels=1, tol=1e-10),
        # many independent fields of uneven sizes at once
        dict(cube, name="batch_64", kind="batch", count=64, size_seed=0),
        # the differentiable solve: forward and adjoint
        dict(cube, name="adjoint_256", kind="adjoint", nx=256, ny=256, nz=256, density="noisy", options="bench",
             levels=5, box="2,2,2", tol=1e-10),
        # the acceleration of a potential, as a particle or gas step takes it after the solve
        dict(cube, name="gravity_256", kind="gravity", nx=256, ny=256, nz=256, density="blobs"),
    ]


def _extents(rng, lo, hi, axes):
    """Extents around one size in [lo, hi] (spread over its logarithm): multiples of a common power of
    two, so that the level rule gives a hierarchy with a small coarsest level."""
    e = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    k = max(2, int(math.log2(e / 4.0)))
    m = e / 2 ** k
    return [2 ** k * max(2, round(m * rng.uniform(0.75, 1.2))) for _ in range(axes)]


def draw(rng):
    case = dict(kind="solve", bc="ddd", box="1,1,1", precision="mixed", options="default", levels=0, tol=1e-8,
                where="device")
    what = rng.choice(["small", "solve", "solve", "host", "large", "periodic", "fp64", "gsrb", "flat", "relax",
                       "batch", "adjoint", "gravity"])
    sizes = {"small": (24, 64), "solve": (48, 256), "host": (48, 256), "large": (200, 400), "periodic": (64, 384),
             "fp64": (32, 192), "gsrb": (32, 256), "adjoint": (32, 256)}
    if what in sizes:
        nx, ny, nz = _extents(rng, *sizes[what], 3)
        case.update(nx=nx, ny=ny, nz=nz, density="blobs")
    if what in ("solve", "gsrb"):
        case["bc"] = rng.choice(["ddd", "pdd", "dpd", "ddp", "ppd"])
    if what == "solve":
        case["options"] = rng.choice(["default", "bench", "rkl1"])
    elif what == "host":
        case["where"] = "host"
    elif what == "large":
        case.update(options="bench", density=rng.choice(["blobs", "noisy"]))
    elif what == "periodic":
        case.update(options=rng.choice(["default", "bench"]), bc="ppp", density="grf")
    elif what == "fp64":
        case.update(options=rng.choice(["default", "bench"]), precision="fp64", tol=1e-10,
                    bc=rng.choice(["ddd", "dpd"]))
    elif what == "gsrb":
        case["options"] = "gsrb"
    elif what == "flat":
        nx, ny = _extents(rng, 64, 2048, 2)
        case.update(nx=nx, ny=ny, nz=0, density="blobs", bc=rng.choice(["dd", "pd"]),
                    options=rng.choice(["default", "bench"]))
    elif what == "relax":
        e = rng.uniform(16, 64)
        nx, ny, nz = (int(e * rng.uniform(0.8, 1.2)) for _ in range(3))
        case.update(nx=nx, ny=ny, nz=nz, density="blobs", levels=1, precision=rng.choice(["fp64", "mixed"]))
    elif what == "batch":
        case.update(kind="batch", count=int(math.exp(rng.uniform(math.log(4), math.log(64)))),
                    size_seed=rng.randrange(1000))
    elif what == "adjoint":
        case.update(kind="adjoint", density="noisy", options=rng.choice(["default", "bench"]), tol=1e-10)
    elif what == "gravity":
        nx, ny, nz = (max(8, int(math.exp(rng.uniform(math.log(24), math.log(320))))) for _ in range(3))
        case.update(kind="gravity", nx=nx, ny=ny, nz=nz, density="blobs", bc=rng.choice(["ddd", "ppp", "dpd"]))
    if case["kind"] != "batch":         # cells of nearly the same width along every axis
        n = [case[a] for a in ("nx", "ny", "nz") if case[a]]
        case["box"] = ",".join("%.3g" % (v / max(n) * rng.uniform(0.9, 1.1)) for v in n)
    return case


# ---- inputs, made on the device ---------------------------------------------------------------

def _geometry(case):
    """Shape (nz, ny, nx) or (ny, nx), and the box (lo, hi) centred on the origin, in x, y (, z) order."""
    axes = 3 if case["nz"] else 2
    ext = [float(v) for v in case["box"].split(",")][:axes]
    shape = (case["nz"], case["ny"], case["nx"])[3 - axes:]
    return shape, tuple(-0.5 * e for e in ext), tuple(0.5 * e for e in ext)


def _axes(shape, lo, hi):
    """Cell centres along x, y (, z)."""
    n = shape[::-1]
    return [lo[d] + (torch.arange(n[d], dtype=torch.float64, device="cuda") + 0.5) * ((hi[d] - lo[d]) / n[d])
            for d in range(len(n))]


def _at(v, d, dims):
    """The coordinates `v` of axis d, broadcast in a C-ordered array of `dims` axes (x last)."""
    return v.reshape([-1 if a == dims - 1 - d else 1 for a in range(dims)])


def _faces(fn, shape, lo, hi, bc):
    """fn at the centres of the boundary faces, -x, +x, -y, +y (, -z, +z); nothing on periodic axes."""
    dims, out = len(shape), []
    xs = _axes(shape, lo, hi)
    for d in range(dims):
        for side in (lo[d], hi[d]):
            if bc[d] == "p":
                out.append(None)
                continue
            at = [_at(torch.full((1,), side, dtype=torch.float64, device="cuda") if a == d else xs[a], a, dims)
                  for a in range(dims)]
            full = fn(at)
            out.append(full.squeeze(dims - 1 - d).contiguous())
    return out


def _sphere(case, rng, shape, lo, hi):
    """A uniform sphere near the middle of the box and its potential on the faces (4 pi G = 1)."""
    dims = len(shape)
    c = [rng.uniform(-0.04, 0.04) * (hi[d] - lo[d]) for d in range(dims)]
    R, rho0 = rng.uniform(0.11, 0.14) * min(hi[d] - lo[d] for d in range(dims)), rng.uniform(0.5, 2.0)
    xs = _axes(shape, lo, hi)
    r2 = sum(_at((xs[d] - c[d]) ** 2, d, dims) for d in range(dims))
    rho = torch.where(r2 <= R * R, rho0, 0.0).to(torch.float64)
    pot = lambda at: -rho0 * R ** 3 / 3.0 / torch.sqrt(sum((at[d] - c[d]) ** 2 for d in range(dims)))
    return rho, _faces(pot, shape, lo, hi, case["bc"])


def _blobs(case, rng, shape, lo, hi):
    """One to four Gaussian blobs and the potential of their total mass on the faces."""
    dims = len(shape)
    ext = [hi[d] - lo[d] for d in range(dims)]
    xs = _axes(shape, lo, hi)
    rho = torch.zeros(shape, dtype=torch.float64, device="cuda")
    for _ in range(rng.randint(1, 4)):
        c = [lo[d] + rng.uniform(0.25, 0.75) * ext[d] for d in range(dims)]
        sig, amp = rng.uniform(0.05, 0.2), rng.uniform(0.5, 2.0)
        part = amp
        for d in range(dims):
            part = part * _at(torch.exp(-(xs[d] - c[d]) ** 2 / (2 * sig * sig)), d, dims)
        rho += part
    total = float(rho.sum())
    cm = [float((rho * _at(xs[d], d, dims)).sum()) / total for d in range(dims)]
    M = total * math.prod(ext[d] / shape[dims - 1 - d] for d in range(dims))
    if dims == 3:
        pot = lambda at: -M / (4 * math.pi) / torch.sqrt(sum((at[d] - cm[d]) ** 2 for d in range(3)))
    else:
        pot = lambda at: M / (4 * math.pi) * torch.log(sum((at[d] - cm[d]) ** 2 for d in range(2)))
    return rho, _faces(pot, shape, lo, hi, case["bc"])


def _grf(case, rng, shape, lo, hi):
    """A periodic Gaussian random field, P(k) ~ |k|^-3, zero mean and unit rms."""
    gen = torch.Generator(device="cuda").manual_seed(rng.randrange(2 ** 31))
    wk = torch.fft.rfftn(torch.randn(shape, dtype=torch.float64, device="cuda", generator=gen))
    k2 = 0.0
    for a, n in enumerate(shape):
        f = torch.fft.rfftfreq(n, device="cuda") if a == len(shape) - 1 else torch.fft.fftfreq(n, device="cuda")
        k2 = k2 + ((f.to(torch.float64) * n) ** 2).reshape([-1 if b == a else 1 for b in range(len(shape))])
    amp = torch.where(k2 > 0, k2.clamp_min(1.0) ** -0.75, 0.0)
    rho = torch.fft.irfftn(wk * amp, s=shape)
    rho -= rho.mean()
    return (rho / rho.square().mean().sqrt()).contiguous(), None


def _noisy(case, rng, shape, lo, hi):
    rho, faces = _sphere(case, rng, shape, lo, hi)
    gen = torch.Generator(device="cuda").manual_seed(rng.randrange(2 ** 31))
    return rho + 0.1 * torch.randn(shape, dtype=torch.float64, device="cuda", generator=gen), faces


DENSITY = {"sphere": _sphere, "noisy": _noisy, "blobs": _blobs, "grf": _grf}


def _inputs(case, seed):
    """(density, faces) of a case with a shape of its own."""
    rng = random.Random("%d %s" % (seed, case["density"]))
    return DENSITY[case["density"]](case, rng, *_geometry(case))


def _weights(case, seed):
    """The loss weights of an adjoint case."""
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    return torch.rand(_geometry(case)[0], dtype=torch.float64, device="cuda", generator=gen)


def _grid(case, faces):
    shape, lo, hi = _geometry(case)
    bc = [sg.PERIODIC if b == "p" else sg.DIRICHLET for b in case["bc"]]
    g = (sg.Grid if len(shape) == 3 else sg.Grid2D)(shape, lo, hi, bc, precision=case["precision"])
    if OPTIONS[case["options"]]:
        g.set_options(**OPTIONS[case["options"]])
    if faces is not None:
        on_host = len(shape) == 2       # a 2D grid takes its four face lines from the host
        g.set_boundary([f if f is None or not on_host else f.cpu().numpy() for f in faces])
    return g


def _batch_members(case, seed):
    """The member cases of a batch: edges from {32, 64, 96, 128}, the same for every seed."""
    sizes = random.Random(case["size_seed"])
    for i in range(case["count"]):
        n = sizes.choice((32, 64, 96, 128))
        yield dict(case, kind="solve", nx=n, ny=n, nz=n, density="blobs"), seed * 1000 + i


def _field(case, seed):
    """A potential to differentiate: smooth, of order one, with the faces that its box has."""
    rho, faces = _inputs(case, seed)
    return (-rho).contiguous(), faces


def prepare(case, seed):
    if case["kind"] == "batch":
        members = list(_batch_members(case, seed))
        made = [_inputs(c, s) for c, s in members]
        return {"case": case, "grids": [_grid(c, f) for (c, _), (_, f) in zip(members, made)],
                "rho": [r for r, _ in made], "phi": [torch.empty_like(r) for r, _ in made]}
    if case["kind"] == "gravity":
        phi, faces = _field(case, seed)
        return {"case": case, "grid": _grid(case, faces), "phi": phi,
                "g": torch.empty((3,) + tuple(phi.shape), dtype=torch.float64, device="cuda")}
    rho, faces = _inputs(case, seed)
    state = {"case": case, "grid": _grid(case, faces)}
    if case["kind"] == "adjoint":
        return dict(state, rho=rho.requires_grad_(True), w=_weights(case, seed))
    if case["where"] == "host":
        rho = rho.cpu().pin_memory()
    return dict(state, rho=rho, phi=torch.empty(rho.shape, dtype=rho.dtype, device=rho.device,
                                                pin_memory=case["where"] == "host"))


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        for g, rho in zip(state["grids"], state["rho"]):
            g.set_density(rho, four_pi_G=1.0)
        sg.solve_batch(state["grids"], tol=case["tol"])
        return [g.potential(phi) for g, phi in zip(state["grids"], state["phi"])]
    if case["kind"] == "gravity":
        return state["grid"].gravity(state["g"], phi=state["phi"])
    if case["kind"] == "adjoint":
        rho = state["rho"]
        rho.grad = None
        phi = sg.solve(rho, state["grid"], tol=case["tol"], levels=case["levels"])
        phi.backward(state["w"])
        return [phi.detach(), rho.grad]
    g = state["grid"]
    g.set_density(state["rho"], four_pi_G=1.0)
    g.solve(tol=case["tol"], levels=case["levels"])
    return g.potential(state["phi"])


def work(case):
    """Bytes: the density read and the potential written (the weights read and the gradient written, for
    an adjoint; three components written, for an acceleration).  Flops: the smoothing that the options ask
    for (twelve a cell and stage on every level) times the typical number of V-cycles."""
    if case["kind"] == "batch":
        parts = [work(c) for c, _ in _batch_members(case, 0)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    cells = case["nx"] * case["ny"] * max(1, case["nz"])
    if case["kind"] == "gravity":
        return {"bytes": 32.0 * cells, "flops": 12.0 * cells}
    o = OPTIONS[case["options"]]
    stages = (o.get("n_pre", 2) + o.get("n_post", 1)) * (1 if case["options"] == "gsrb" else o.get("s_smooth", 3))
    cycles = CYCLES[case["options"]] * -math.log10(case["tol"]) / 8.0
    below = 1.0 / 7.0 if case["nz"] else 1.0 / 3.0          # the cells of all coarser levels
    if case["levels"] == 1:
        stages, below, cycles = 6 * max(case["nx"], case["ny"], case["nz"]), 0.0, 1
    both = 2 if case["kind"] == "adjoint" else 1
    return {"bytes": 16.0 * cells * both, "flops": 12.0 * cells * (1 + below) * stages * cycles * both}


# ---- the same results in 64 bits, without the solver ------------------------------------------

def _basis(n, h, periodic):
    """Orthonormal eigenvectors (rows) and eigenvalues of the cell-centred second difference along one axis:
    sines about the walls (the ghost is minus the cell) or the real Fourier modes."""
    i = torch.arange(n, dtype=torch.float64, device="cuda") + 0.5
    if not periodic:
        k = torch.arange(1, n + 1, dtype=torch.float64, device="cuda")
        V = torch.sin(math.pi * k[:, None] * i[None, :] / n) * math.sqrt(2.0 / n)
        V[-1] *= math.sqrt(0.5)
        return V, -(4.0 / h ** 2) * torch.sin(math.pi * k / (2 * n)) ** 2
    k = torch.arange(n, dtype=torch.float64, device="cuda")
    w = torch.minimum(k, n - k)
    V = torch.where((k <= n // 2)[:, None], torch.cos(2 * math.pi * w[:, None] * (i[None, :] - 0.5) / n),
                    torch.sin(2 * math.pi * w[:, None] * (i[None, :] - 0.5) / n))
    V = V / V.square().sum(1, keepdim=True).sqrt()
    return V, -(4.0 / h ** 2) * torch.sin(math.pi * w / n) ** 2


def _along(V, x, axis):
    return torch.movedim(torch.tensordot(V, x, dims=([1], [axis])), 0, axis)


def _direct(case, rhs, faces):
    """The solution of L phi = rhs under the ghost rules, by diagonalising L."""
    shape, lo, hi = _geometry(case)
    dims = len(shape)
    x = rhs.clone()
    bases, lam = [], 0.0
    for d in range(dims):
        a, n = dims - 1 - d, shape[dims - 1 - d]
        h = (hi[d] - lo[d]) / n
        if case["bc"][d] == "d" and faces is not None:
            x.select(a, 0).sub_(2.0 / h ** 2 * faces[2 * d])
            x.select(a, n - 1).sub_(2.0 / h ** 2 * faces[2 * d + 1])
        V, ev = _basis(n, h, case["bc"][d] == "p")
        bases.append((a, V))
        lam = lam + ev.reshape([-1 if b == a else 1 for b in range(dims)])
    if set(case["bc"]) == {"p"}:
        x -= x.mean()
    for a, V in bases:
        x = _along(V, x, a)
    x = torch.where(lam < 0, x / torch.where(lam < 0, lam, -1.0), 0.0)
    for a, V in bases:
        x = _along(V.T.contiguous(), x, a)
    return x


def _acceleration(case, phi, faces):
    """-grad phi to fourth order; past a wall phi continues as the odd reflection about the face value."""
    shape, lo, hi = _geometry(case)
    dims = len(shape)
    out = []
    for d in range(dims):
        a, n = dims - 1 - d, shape[dims - 1 - d]
        if case["bc"][d] == "p":
            ext = torch.cat([phi.narrow(a, n - 2, 2), phi, phi.narrow(a, 0, 2)], a)
        else:
            f0, f1 = (faces[2 * d + s].unsqueeze(a) for s in (0, 1))
            ext = torch.cat([2 * f0 - phi.narrow(a, 0, 2).flip(a), phi, 2 * f1 - phi.narrow(a, n - 2, 2).flip(a)], a)
        p = [ext.narrow(a, s, n) for s in range(5)]
        out.append(-(8.0 * (p[3] - p[1]) - (p[4] - p[0])) / (12.0 * (hi[d] - lo[d]) / n))
    return torch.stack(out)


def exact(case, seed):
    if case["kind"] == "batch":
        return [_direct(c, *_inputs(c, s)) for c, s in _batch_members(case, seed)]
    if case["kind"] == "gravity":
        return _acceleration(case, *_field(case, seed))
    phi = _direct(case, *_inputs(case, seed))
    if case["kind"] == "adjoint":
        return [phi, _direct(case, _weights(case, seed), None)]
    return phi
