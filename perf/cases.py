"""What a user of this framework has it do, as cases that can be timed and compared.

Kinds of case
  step      a single run (2D, or 3D with Fourier planes) advances ``steps`` time steps and its fields
            are read: the loop of a simulation program (Solver.step, Solver.get_into)
  ensemble  independent 2D runs of uneven meshes advance together and every run's fields are read
            (Batch.step, Batch.get)
  march     an ensemble on one mesh marches the equilibrium system in pseudo-time with the per-run
            exit, as the data generation of the learned warm start does
            (Batch.run_to_equilibrium, Batch.get)
  solve     one Helmholtz solve on a user's right-hand side, host arrays (Solver.solve_helmholtz)
  static    the allocation-free solve on device arrays (fdm_solve_static)
  train     epochs of Adam training of the warm-start network (NeuralOperator.train)

Meshes, plane counts, precisions and options are those of this repository's workloads, tests and
benchmark and sizes between them; the physics is that of its small parity runs (a resolved interface,
moderate ratios, a larger mobility and time step), in which the FP32 rounding of the pressure and
velocity stays small beside their values over a few steps.  FP32 (mixed) results are returned in FP32.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2305_09020_gb300 import native

FIELDS = native.PF_FIELD_V | native.PF_FIELD_PHI | native.PF_FIELD_P | native.PF_FIELD_U
EQ_FIELDS = native.PF_FIELD_V | native.PF_FIELD_PHI


def _step(name, ex, ey, order, nz, mixed, steps, wall="electrode", model="full", theta=90.0, graded=False):
    return dict(name=name, kind="step", ex=ex, ey=ey, order=order, nz=nz, mixed=mixed, steps=steps, wall=wall,
                model=model, theta=theta, graded=graded)


def listed():
    return [
        # the smallest run, read after every step: launches and latency (the 2D droplet's mesh, FP64,
        # the default precision)
        _step("droplet2d_fp64", 8, 4, 6, 1, False, 1),
        # the same mesh in mixed precision
        _step("droplet2d_mixed", 8, 4, 6, 1, True, 2),
        # 2D with a graded wall layer, an odd node count in x (no 16-byte rows), contact angle 60 degrees
        _step("film2d_fp64", 15, 6, 7, 1, False, 10, theta=60.0, graded=True),
        # the ordinary 3D run (the 3D droplet's mesh), FP64 and mixed
        _step("droplet3d_fp64", 16, 8, 8, 64, False, 4),
        _step("droplet3d_mixed", 16, 8, 8, 64, True, 2),
        # the electrode array: patches on the wall, 120 planes (mixed radix), the equilibrium system
        _step("array3d_fp64", 20, 6, 12, 120, False, 2, wall="patches", model="equilibrium"),
        # the large 3D run (13.2 million values per field)
        _step("layers3d_mixed", 32, 16, 10, 256, True, 2),
        # a parameter study: runs of uneven meshes side by side
        dict(name="ensemble2d_fp64", kind="ensemble", runs=48, mixed=False, steps=10),
        # training data of the warm start: one mesh, equilibrium system, per-run exit, FP64
        dict(name="march2d_fp64", kind="march", runs=128, ex=8, ey=4, order=6, mixed=False, steps=40),
        # one solve from a host program (pressure set, one Fourier mode)
        dict(name="helmholtz_fp64", kind="solve", ex=16, ey=8, order=8, nz=64, mixed=False, bcset=native.PF_BCSET_P),
        # a solve inside a caller's own device loop
        dict(name="static_fp64", kind="static", ex=16, ey=8, order=8, planes=64),
        # the warm-start network
        dict(name="operator_train", kind="train", samples=256, batch=64, epochs=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 7 + ["ensemble", "march", "solve", "static", "train"])
    mixed = rng.random() < 0.5
    order = rng.randint(4, 12)
    if kind == "step":
        if rng.random() < 0.3:      # 2D
            ex = rng.randint(4, 24)
            return dict(kind=kind, ex=ex, ey=max(2, ex // 2), order=order, nz=1, mixed=mixed,
                        steps=rng.choice([1, 2] if mixed else [1, 5, 10, 20]),
                        wall=rng.choice(["electrode", "neumann_top"] if mixed else ["electrode", "neumann_top", "patches"]),
                        model="full", theta=rng.choice([90.0, 60.0, 75.0]), graded=rng.random() < 0.3)
        ex, nz = rng.randint(4, 24), rng.choice([8, 16, 24, 30, 32, 48, 64, 96, 100, 120, 128])
        ey = max(2, ex // 2)
        values = ex * order * (ey * order + 1) * nz
        most = 2.2e6 if mixed else 1.1e6
        if values > most:
            ex = max(4, int(ex * math.sqrt(most / values)))
            ey = max(2, ex // 2)
        return dict(kind=kind, ex=ex, ey=ey, order=order, nz=nz, mixed=mixed, steps=rng.choice([1, 2] if mixed else [1, 2, 4]),
                    wall=rng.choice(["electrode", "neumann_top"]), model=rng.choice(["full", "full", "equilibrium"]),
                    theta=rng.choice([90.0, 90.0, 60.0]), graded=rng.random() < 0.3)
    if kind == "ensemble":
        return dict(kind=kind, runs=_log_int(rng, 4, 40), mixed=mixed, steps=2 if mixed else rng.choice([5, 10, 20]))
    if kind == "march":
        return dict(kind=kind, runs=_log_int(rng, 16, 256), ex=rng.choice([8, 12, 16]), ey=rng.choice([4, 6]),
                    order=rng.randint(4, 8), mixed=mixed, steps=rng.choice([5, 10] if mixed else [10, 20, 40]))
    if kind == "solve":
        ex = rng.randint(4, 20)
        return dict(kind=kind, ex=ex, ey=max(2, ex // 2), order=min(order, 10), nz=rng.choice([1, 8, 30, 64]), mixed=mixed,
                    bcset=rng.choice([native.PF_BCSET_V, native.PF_BCSET_P, native.PF_BCSET_U]))
    if kind == "static":
        ex = rng.randint(3, 24)
        ey = max(1, ex // 2)
        n2 = ex * order * (ey * order + 1)
        return dict(kind=kind, ex=ex, ey=ey, order=order, planes=max(1, min(_log_int(rng, 1, 128), (1 << 20) // n2)))
    return dict(kind=kind, samples=_log_int(rng, 128, 512), batch=rng.choice([32, 48, 64]), epochs=rng.randint(2, 10))


# ---- inputs --------------------------------------------------------------------------------------
def _breaks(c):
    yb = np.linspace(0.0, 1.0, c["ey"] + 1)
    if c.get("graded"):     # small elements at the wall and the open side
        yb = 0.5 * (1.0 - np.cos(np.pi * yb))
    return np.linspace(0.0, c["ex"] / c["ey"], c["ex"] + 1), yb


def _drop(rng, x, y, z, lx, lz, eta):
    """tanh profile of a drop near the wall, [z][y][x] on the GPU (periodic in x and z)."""
    x, y, z = (torch.as_tensor(a, dtype=torch.float64, device="cuda") for a in (x, y, z))
    r0 = rng.uniform(0.25, 0.35)
    dx = torch.remainder(x - rng.uniform(0.4, 0.6) * lx + 0.5 * lx, lx) - 0.5 * lx
    r2 = (dx ** 2)[None, None, :] + ((y - rng.uniform(0.2, 0.5)) ** 2)[None, :, None]
    if len(z) > 1:
        dz = torch.remainder(z - rng.uniform(0.4, 0.6) * lz + 0.5 * lz, lz) - 0.5 * lz
        r2 = r2 + (dz ** 2)[:, None, None]
    return torch.tanh((r0 - torch.sqrt(r2)) / (math.sqrt(2.0) * eta)).cpu().numpy()


def _flow(rng, x, y, z, lx, lz):
    """A smooth initial velocity that vanishes on the wall, three blocks [z][y][x]."""
    x, y, z = (torch.as_tensor(a, dtype=torch.float64, device="cuda") for a in (x, y, z))
    X, Y, Z = x[None, None, :] * (2 * math.pi / lx), y[None, :, None], z[:, None, None] * (2 * math.pi / lz)
    a = [rng.uniform(0.3, 0.6) for _ in range(3)]
    b = [rng.uniform(0.0, 2 * math.pi) for _ in range(3)]
    ux = a[0] * Y * (2 - Y) * torch.cos(X + b[0]) * (1 + 0.5 * torch.cos(Z))
    uy = a[1] * Y * Y * torch.sin(X + b[1]) * (1 + 0.5 * torch.sin(Z))
    uz = a[2] * Y * (2 - Y) * torch.sin(Z + b[2]) * (1 + 0.5 * torch.cos(X)) if len(z) > 1 else torch.zeros_like(ux)
    shape = (len(z), len(y), len(x))
    return torch.stack([u.expand(shape) for u in (ux, uy, uz)]).cpu().numpy()


def _vbc(c, rng, lx):
    v = rng.uniform(1.5, 2.5)
    wall = c.get("wall", "electrode")
    if wall == "patches":       # alternating stripes, an open top
        n = 5
        pats = tuple((i * lx / n, (i + 0.5) * lx / n, v if i % 2 == 0 else -v) for i in range(n))
        return dict(bottom_kind=native.PF_BC_PATCHES, top_kind=native.PF_BC_NEUMANN, v_bottom=0.0, v_top=0.0, patches=pats)
    top = native.PF_BC_NEUMANN if wall == "neumann_top" else native.PF_BC_DIRICHLET
    return dict(bottom_kind=native.PF_BC_DIRICHLET, top_kind=top, v_bottom=v, v_top=0.0, patches=())


def _solver(c, seed, state):
    rng = np.random.default_rng(seed)
    xb, yb = _breaks(c)
    order, nz, lz = c["order"], c["nz"], 1.0
    x, y = native.nodes_1d(xb, order, True), native.nodes_1d(yb, order, False)
    z = np.arange(nz) * (lz / nz)
    fluid = dict(rho1=2.0, rho2=1.0, mu1=0.2, mu2=0.1, eps1=rng.uniform(1.8, 2.2), eps2=1.0, sigma=1.0, eta=0.1,
                 gamma1=1e-2, theta_s_deg=c.get("theta", 90.0))
    scheme = dict(dt=5e-4, bdf=2, precision=native.PF_MIXED if c["mixed"] else native.PF_FP64,
                  model=native.PF_MODEL_EQUILIBRIUM if c.get("model") == "equilibrium" else native.PF_MODEL_FULL)
    u0 = None if c.get("model") == "equilibrium" else _flow(rng, x, y, z, xb[-1], lz)
    state["stream"] = torch.cuda.Stream()
    return native.Solver(xb, yb, order, nz, lz, fluid, _vbc(c, rng, xb[-1]), scheme,
                         _drop(rng, x, y, z, xb[-1], lz, fluid["eta"]), u0, stream=state["stream"].cuda_stream)


def _runs(c, rng):
    """Descriptors of independent 2D runs: uneven meshes (ensemble) or one mesh (march)."""
    runs, phis = [], []
    for i in range(c["runs"]):
        if c["kind"] == "ensemble":
            ex = 4 + 2 * ((7 * i) % 9)      # 4 .. 20 elements, orders 4 .. 10: many meshes
            ey, order = ex // 2, 4 + (5 * i) % 7
        else:
            ex, ey, order = c["ex"], c["ey"], c["order"]
        eta, march = 0.04, c["kind"] == "march"
        mesh = SimpleNamespace(ex=ex, ey=ey, order=order, nz=1, lz=1.0, xb=np.linspace(0.0, 2.0, ex + 1),
                               yb=np.linspace(0.0, 1.0, ey + 1))
        fluid = SimpleNamespace(rho1=1.0, rho2=1.0, mu1=1.0, mu2=1.0, eps1=rng.uniform(1.5, 4.0), eps2=1.0, sigma=1.0,
                                eta=eta, gamma1=3e-3, theta_s_deg=90.0)
        vbc = SimpleNamespace(bottom_kind=native.PF_BC_DIRICHLET, top_kind=native.PF_BC_DIRICHLET,
                              v_bottom=rng.uniform(0.0, 1.0), v_top=0.0)
        scheme = SimpleNamespace(dt=1e-3, bdf=2, S=0.0, nu_m=0.0, rho0=0.0, eps0=0.0, equilibrium=march)
        runs.append(SimpleNamespace(mesh=mesh, fluid=fluid, vbc=vbc, scheme=scheme))
        x, y = native.nodes_1d(mesh.xb, order, True), native.nodes_1d(mesh.yb, order, False)
        r0 = rng.uniform(0.25, 0.35)
        r = np.sqrt((x[None, :] - 1.0) ** 2 + y[:, None] ** 2)
        phis.append(np.tanh((r0 - r) / (math.sqrt(2.0) * eta)))
    return runs, phis


DIMS, GRID, BOX = [3, 128, 384, 128 * 64], (128, 64), (0.0, 2.0, 0.0, 1.0)   # the warm-start network


def prepare(case, seed):
    c, rng = case, np.random.default_rng(seed)
    s = {"case": c}
    if c["kind"] == "step":
        s["solver"] = _solver(c, seed, s)
        s["mask"] = EQ_FIELDS if c["model"] == "equilibrium" else FIELDS
        s["blocks"] = 2 if c["model"] == "equilibrium" else 6
        s["host"] = torch.empty(s["blocks"] * s["solver"].n, dtype=torch.float64, pin_memory=True)
    elif c["kind"] in ("ensemble", "march"):
        runs, phis = _runs(c, rng)
        s["stream"] = torch.cuda.Stream()
        s["batch"] = native.Batch(runs, native.PF_MIXED if c["mixed"] else native.PF_FP64,
                                  stream=s["stream"].cuda_stream, phi0_list=phis)
        s["taken"] = 0
    elif c["kind"] == "solve":
        s["solver"] = _solver(dict(c, model="equilibrium"), seed, s)
        nz = c["nz"]
        s["mode"] = 0 if nz == 1 else int(rng.integers(1, nz // 2))
        s["lam"] = float(rng.uniform(0.5, 50.0))
        s["rhs"] = rng.standard_normal((1 if s["mode"] == 0 else 2, s["solver"].ny, s["solver"].nx))
    elif c["kind"] == "static":
        xb, yb = _breaks(c)
        Kx, Mx = native.operators_1d(xb, c["order"], True)
        Ky, My = native.operators_1d(yb, c["order"], False)
        d = np.zeros(len(My), dtype=np.uint8)
        d[-1] = 1                       # natural on the wall, Dirichlet on the open side
        (Sx, Lx), (Sy, Ly) = native.fdm_1d(Kx, Mx), native.fdm_1d(Ky, My, d)
        rhs, shift = _static_inputs(c, seed, len(Mx), len(My))
        rhs = rhs * (torch.as_tensor(My, device="cuda")[:, None] * torch.as_tensor(Mx, device="cuda")[None, :])
        up = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")  # noqa: E731
        s.update(nx=len(Mx), ny=len(My), tables=[up(Sx), up(Sx.T), up(Lx), up(Sy), up(Sy.T), up(Ly)],
                 shift=shift, rhs=rhs.contiguous(), out=torch.empty_like(rhs))
    else:
        x, y = native.nodes_1d(np.linspace(0.0, 2.0, 9), 6, True), native.nodes_1d(np.linspace(0.0, 1.0, 5), 6, False)
        v, e, r = rng.uniform(0, 3, c["samples"]), np.exp(rng.uniform(math.log(2), math.log(20), c["samples"])), \
            rng.uniform(0.15, 0.35, c["samples"])
        s["feat"] = np.stack([v, e, 0.5 * math.pi * r ** 2], axis=1)
        stretch = (1 + 0.05 * v)[:, None, None]
        d = np.sqrt(((x - 1.0)[None, None, :] * stretch) ** 2 + (y[None, :, None] / stretch) ** 2)
        s["target"] = np.tanh((r[:, None, None] - d) / (math.sqrt(2.0) * 0.02)).reshape(c["samples"], -1)
        s["stream"] = torch.cuda.Stream()
        s["net"] = native.NeuralOperator(DIMS, s["feat"].mean(0), s["feat"].std(0) + 1e-12, GRID, BOX, x, y,
                                         seed=seed & 0x7FFFFFFF, stream=s["stream"].cuda_stream)
    return s


def _static_inputs(c, seed, nx, ny):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    rhs = torch.randn(c["planes"], ny, nx, dtype=torch.float64, device="cuda", generator=g)
    shift = 0.5 + 100.0 * torch.rand(c["planes"], dtype=torch.float64, device="cuda", generator=g)
    return rhs, shift


def run(s):
    c = s["case"]
    if c["kind"] == "step":
        # one block [field][z][y][x] per field; a mixed run's fields go on in FP32 on the GPU
        s["solver"].step(c["steps"])
        s["solver"].get_into(s["mask"], s["host"].numpy())
        host = s["host"].view(s["blocks"], -1)
        if c["mixed"]:
            host = host.to("cuda").float()
        return {"V": host[0], "phi": host[1]} if s["blocks"] == 2 else \
            {"V": host[0], "phi": host[1], "P": host[2], "u": host[3:]}
    if c["kind"] in ("ensemble", "march"):
        b = s["batch"]
        out = {}
        if c["kind"] == "march":
            s["taken"] += c["steps"]
            out["exit"] = b.run_to_equilibrium(1e-3, s["taken"], c["steps"])
        else:
            b.step(c["steps"])
        mask = EQ_FIELDS if c["kind"] == "march" else FIELDS
        per_run = [b.get(r, mask) for r in range(c["runs"])]
        dtype = np.float32 if c["mixed"] else np.float64
        for name, parts in (("V", ("V",)), ("phi", ("phi",)), ("P", ("P",)), ("u", ("ux", "uy"))):
            if parts[0] in per_run[0]:
                out[name] = np.concatenate([f[k].ravel() for f in per_run for k in parts]).astype(dtype, copy=False)
        return out
    if c["kind"] == "solve":
        x = s["solver"].solve_helmholtz(c["bcset"], s["mode"], s["lam"], s["rhs"])
        return x.astype(np.float32) if c["mixed"] else x
    if c["kind"] == "static":
        native.fdm_solve_static(s["nx"], s["ny"], c["planes"], *(t.data_ptr() for t in s["tables"]),
                                s["shift"].data_ptr(), s["rhs"].data_ptr(), s["out"].data_ptr(),
                                torch.cuda.current_stream().cuda_stream)
        return s["out"]
    losses = s["net"].train(s["feat"], s["target"], batch=c["batch"], epochs=c["epochs"], lr=1e-3, seed=3)
    return {"losses": losses.astype(np.float32), "params": s["net"].params().astype(np.float32)}


# ---- the work that a pass cannot do without ------------------------------------------------------
def _fdm_flops(nx, ny, planes):
    return 4.0 * nx * ny * (nx + ny) * planes


def work(case):
    c = case
    if c["kind"] == "step":
        nx, ny, nz = c["ex"] * c["order"], c["ey"] * c["order"] + 1, c["nz"]
        n, w = nx * ny * nz, 4.0 if c["mixed"] else 8.0
        d3, eq = nz > 1, c["model"] == "equilibrium"
        solves = (4 if c["wall"] == "patches" else 3) if eq else ((7 if d3 else 6) + (c["wall"] == "patches"))
        # the two history levels read, the new level written, each solve's right-hand side and
        # solution once; the fields read out in FP64
        fields = 3 * ((4 if d3 else 2) if eq else (12 if d3 else 5)) + 2 * solves
        return {"bytes": c["steps"] * fields * n * w + (2 if eq else 6) * n * 8.0,
                "flops": c["steps"] * solves * _fdm_flops(nx, ny, nz)}
    if c["kind"] in ("ensemble", "march"):
        total = {"bytes": 0.0, "flops": 0.0}
        for i in range(c["runs"]):
            if c["kind"] == "ensemble":
                ex = 4 + 2 * ((7 * i) % 9)
                ey, order = ex // 2, 4 + (5 * i) % 7
            else:
                ex, ey, order = c["ex"], c["ey"], c["order"]
            nx, ny, eq = ex * order, ey * order + 1, c["kind"] == "march"
            n, solves = nx * ny, 3 if eq else 5
            total["bytes"] += c["steps"] * (3 * (2 if eq else 5) + 2 * solves) * n * (4.0 if c["mixed"] else 8.0) + \
                (2 if eq else 6) * n * 8.0
            total["flops"] += c["steps"] * solves * _fdm_flops(nx, ny, 1)
        return total
    if c["kind"] in ("solve", "static"):
        nx, ny = c["ex"] * c["order"], c["ey"] * c["order"] + 1
        planes = c["planes"] if c["kind"] == "static" else 1 if c["nz"] == 1 else 2
        w = 4.0 if c.get("mixed") else 8.0
        return {"bytes": (2.0 * nx * ny * planes + nx * nx + ny * ny) * w, "flops": _fdm_flops(nx, ny, planes)}
    params = sum(a * b + b for a, b in zip(DIMS, DIMS[1:]))
    batches = c["epochs"] * (c["samples"] // c["batch"])
    # per batch: weights, gradients and both moments read and written once; forward and two backward
    # products
    return {"bytes": batches * params * 4.0 * 7.0, "flops": batches * 6.0 * params * c["batch"]}


# ---- plain 64-bit values ---------------------------------------------------------------------------
def _operators(breaks, order, periodic):
    """1D GLL stiffness and diagonal mass of a spectral-element mesh, plain numpy."""
    leg = np.polynomial.legendre.Legendre.basis(order)
    xi = np.concatenate([[-1.0], np.sort(leg.deriv().roots().real), [1.0]])
    for _ in range(3):      # Newton on (1 - x^2) P'(x): full accuracy of the interior nodes
        xi[1:-1] -= leg.deriv()(xi[1:-1]) / leg.deriv(2)(xi[1:-1])
    w = 2.0 / (order * (order + 1) * leg(xi) ** 2)
    p = order + 1
    D = np.zeros((p, p))
    for i in range(p):
        for j in range(p):
            if i != j:
                D[i, j] = leg(xi[i]) / (leg(xi[j]) * (xi[i] - xi[j]))
        D[i, i] = -D[i].sum()
    ref = D.T @ (w[:, None] * D)
    ne = len(breaks) - 1
    n = ne * order + (0 if periodic else 1)
    K, M = np.zeros((n, n)), np.zeros(n)
    for e in range(ne):
        h = breaks[e + 1] - breaks[e]
        ids = (e * order + np.arange(p)) % n
        K[np.ix_(ids, ids)] += (2.0 / h) * ref
        M[ids] += 0.5 * h * w
    return K, M


def _dense_solve(Kx, Mx, Ky, My, free, shifts, f):
    """x = (K + shift M)^-1 M f per plane on the free y nodes, by the symmetric eigenproblems."""
    def basis(K, M):
        r = 1.0 / np.sqrt(M)
        lam, q = np.linalg.eigh(K * r[:, None] * r[None, :])
        return lam, q * r[:, None]
    lx, sx = basis(Kx, Mx)
    ly, sy = basis(Ky[np.ix_(free, free)], My[free])
    out = np.zeros_like(f)
    for p in range(f.shape[0]):
        b = (My[:, None] * Mx[None, :] * f[p])[free]
        out[p, free] = sy @ ((sy.T @ b @ sx) / (ly[:, None] + lx[None, :] + shifts[p])) @ sx.T
    return out


def exact(case, seed):
    """The two solves in 64 bits.  The time steps and the training have none here: a step's plain
    restatement takes far longer than the 20 seconds at these sizes (assembled direct solves per
    Fourier mode), and training rounds its weights to BF16 on every update."""
    c = case
    if c["kind"] not in ("solve", "static"):
        return None
    xb, yb = _breaks(c)
    Kx, Mx = _operators(xb, c["order"], True)
    Ky, My = _operators(yb, c["order"], False)
    ny, nx = len(My), len(Mx)
    if c["kind"] == "static":
        rhs, shift = _static_inputs(c, seed, nx, ny)
        return torch.from_numpy(_dense_solve(Kx, Mx, Ky, My, np.arange(ny - 1), shift.cpu().numpy(), rhs.cpu().numpy()))
    rng = np.random.default_rng(seed)
    mode = 0 if c["nz"] == 1 else int(rng.integers(1, c["nz"] // 2))
    lam = float(rng.uniform(0.5, 50.0))
    f = rng.standard_normal((1 if mode == 0 else 2, ny, nx))
    free = {native.PF_BCSET_V: np.arange(1, ny - 1), native.PF_BCSET_P: np.arange(ny - 1),
            native.PF_BCSET_U: np.arange(1, ny)}[c["bcset"]]
    shift = lam + (2 * math.pi * mode) ** 2
    return _dense_solve(Kx, Mx, Ky, My, free, [shift] * f.shape[0], f).ravel()
