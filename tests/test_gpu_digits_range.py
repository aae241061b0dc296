"""Digit products whose operands are of uneven size: graded meshes, whose eigenbases and mass-weighted
right-hand sides are large at opposite ends, values at constrained nodes, which no solution depends on, and
eigenbases of uncoupled pieces.  Per plane and per row, against extended precision and beside the FMA chains."""
import numpy as np
import pytest

import workloads
from paper_2305_09020_gb300 import native

pytestmark = pytest.mark.gpu

LAM, MODE = 2.5, 1


def _growing(g, n):
    y = np.concatenate([[0.0], np.cumsum(float(g) ** np.arange(n))])
    return y / y[-1]


MESHES = {
    "even": (np.linspace(0.0, 8.0, 9), np.linspace(0.0, 1.0, 9), 6),
    "cosine": (np.linspace(0.0, 2.5, 16), 0.5 * (1.0 - np.cos(np.pi * np.linspace(0.0, 1.0, 7))), 7),
    "2x8": (np.linspace(0.0, 4.0, 9), _growing(2, 8), 6),
    "2x16": (np.linspace(0.0, 4.0, 9), _growing(2, 16), 6),
    "4x11": (np.linspace(0.0, 4.0, 9), _growing(4, 11), 6),
    "graded x": (np.concatenate([-_growing(3, 8)[:0:-1], _growing(3, 8)]), np.linspace(0.0, 1.0, 9), 6),
}


def _factors(xb, yb, K, fixed=(-1,)):
    Kx, Mx = native.operators_1d(xb, K, True)
    Ky, My = native.operators_1d(yb, K, False)
    d = np.zeros(len(My), dtype=np.uint8)
    d[list(fixed)] = 1
    (Sx, Lx), (Sy, Ly) = native.fdm_1d(Kx, Mx), native.fdm_1d(Ky, My, d)
    Lx[np.abs(Lx) < 1e-11] = 0.0
    Ly[np.abs(Ly) < 1e-11] = 0.0
    return Sx, Lx, Sy, Ly, Mx, My


def _reference(b, fac, shift):
    Sx, Lx, Sy, Ly = (a.astype(np.longdouble) for a in fac[:4])
    return np.array([Sy @ ((Sy.T @ pl.astype(np.longdouble) @ Sx) / (Ly[:, None] + Lx[None, :] + np.longdouble(shift))) @ Sx.T
                     for pl in b])


def _errors(x, ref):
    """Relative errors of each plane, and of the worst row and column with a solution in it."""
    d, r = (x.astype(np.longdouble) - ref).astype(np.float64), ref.astype(np.float64)
    plane = max(np.linalg.norm(d[p]) / np.linalg.norm(r[p]) for p in range(len(r)))
    out = [float(plane)]
    for ax in (2, 1):
        n = np.linalg.norm(r, axis=ax)
        out.append(float((np.linalg.norm(d, axis=ax)[n > 0] / n[n > 0]).max()))
    return out


def _within(err, fma):
    """No measure above the FMA chains'.  Where those happen to be exact, four products and a quotient
    that round once each leave 2.5 units of 1.1e-16, and a row or column that is small against the
    intermediate plane may hold a few times that."""
    return all(e <= max(f, 1e-15) for e, f in zip(err, fma))


def _static(fac, b, shift):
    torch = pytest.importorskip("torch")
    Sx, Lx, Sy, Ly, Mx, My = fac
    t = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")  # noqa: E731
    dev = [t(a) for a in (Sx, Sx.T, Lx, Sy, Sy.T, Ly)]
    sh, rhs = t(np.full(len(b), shift)), t(b)
    out = torch.empty_like(rhs)
    native.fdm_solve_static(len(Mx), len(My), len(b), *(x.data_ptr() for x in dev), sh.data_ptr(), rhs.data_ptr(),
                            out.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("scale", [1.0, 1e6, 1e14, 1e200])
@pytest.mark.parametrize("mesh", MESHES)
def test_graded_meshes_and_constrained_nodes(mesh, scale):
    """The pressure set (Dirichlet on the open side), two planes of unlike size, the right-hand side at the
    constrained nodes scaled up: FP64 run by digits and by FMA chains, and the allocation-free solve."""
    xb, yb, K = MESHES[mesh]
    wl = workloads.small3d(ex=len(xb) - 1, ey=len(yb) - 1, order=K, nz=4)
    wl.mesh.xb, wl.mesh.yb = xb, yb
    fac = _factors(xb, yb, K)
    Mx, My = fac[4:]
    f = np.random.default_rng(len(yb)).standard_normal((2, len(My), len(Mx)))
    f[1] *= 1e-9
    f[:, -1] *= scale
    b = (Mx[None, :] * My[:, None]) * f
    shift = LAM + (2 * np.pi * MODE / wl.mesh.lz) ** 2
    ref = _reference(b, fac, shift)
    g = native.from_workload(wl, precision=native.PF_FP64)
    x = g.solve_helmholtz(native.PF_BCSET_P, MODE, LAM, f).reshape(f.shape)
    g.set_variant(native.PF_GEMM_SIMT32, fuse_y=False)
    fma = _errors(g.solve_helmholtz(native.PF_BCSET_P, MODE, LAM, f).reshape(f.shape), ref)
    g.close()
    digits, static = _errors(x, ref), _errors(_static(fac, b, shift), ref)
    print(mesh, scale, "fma", fma, "digits", digits, "static", static)
    assert _within(digits, fma), (digits, fma)
    assert _within(static, fma), (static, fma)


@pytest.mark.parametrize("ratio", [1.0, 1e10, 1e-10, 1e30])
def test_static_solve_of_uncoupled_pieces(ratio):
    """A Dirichlet node inside the mesh parts it into two pieces: the eigenbasis has zeros between them, and
    a right-hand side of another size in one piece leaves the other's solution as exact as it was."""
    xb, yb, K = np.linspace(0.0, 4.0, 9), np.linspace(0.0, 1.0, 9), 6
    fac = _factors(xb, yb, K, fixed=(4 * K, -1))
    Mx, My = fac[4:]
    f = np.random.default_rng(5).standard_normal((2, len(My), len(Mx)))
    f[:, :4 * K] *= ratio
    b = (Mx[None, :] * My[:, None]) * f
    ref = _reference(b, fac, LAM)
    x = _static(fac, b, LAM)
    for rows in (slice(0, 4 * K), slice(4 * K + 1, None)):
        d, r = (x[:, rows] - ref[:, rows]).astype(np.float64), ref[:, rows].astype(np.float64)
        assert np.linalg.norm(d) <= 1e-14 * np.linalg.norm(r)     # sums of 49 terms, four products


@pytest.mark.parametrize("meshes", [[(8, 4, 6)] * 3, [(8, 4, 6), (7, 5, 5), (8, 4, 6)]])
def test_runs_of_an_ensemble_freeze_at_different_steps(meshes):
    """Planes of 28 nodes and up, whose 128-row units hold frozen and live runs: every run stops at the step, and
    with the fields, that the FMA transforms give it."""
    runs = []
    for i, (ex, ey, K) in enumerate(meshes):
        wl = workloads.small2d(ex=ex, ey=ey, order=K)
        wl.fluid.eps1, wl.vbc.v_bottom, wl.scheme.equilibrium = 2.0 + 4.0 * i, 0.5 + i, True
        runs.append(wl)
    alone = []
    for wl in runs:
        h = native.from_workload(wl, precision=native.PF_FP64)
        r = []
        for _ in range(12):
            h.step(1)
            r.append(h.diagnostics()[6])
        h.close()
        alone.append(r)
    at = sorted(r[5] for r in alone)
    tol = float(np.sqrt(at[0] * at[1]))
    got = []
    for gemm in (None, native.PF_GEMM_SIMT32):
        b = native.Batch(runs, precision=native.PF_FP64)
        if gemm is not None:
            b.set_variant(gemm, fuse_y=False)
        steps = b.run_to_equilibrium(tol=tol, max_steps=12, check_every=5)
        got.append((list(steps), [b.get(i, native.PF_FIELD_V | native.PF_FIELD_PHI) for i in range(len(runs))]))
        b.close()
    assert got[0][0] == got[1][0] and len(set(got[0][0])) > 1, got
    for a, c in zip(got[0][1], got[1][1]):
        for k in a:
            assert np.linalg.norm(a[k] - c[k]) <= 1e-12 * np.linalg.norm(c[k]), k
