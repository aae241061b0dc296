"""The FP64 transforms by digit products on the tensor cores (the default of an FP64 run) against
extended precision, beside the FMA chains of the CUDA-core variants."""
import numpy as np
import pytest

import workloads
from paper_2305_09020_gb300 import native

pytestmark = pytest.mark.gpu

# (ex, ey, K): one stage of 32 and remainders, both column-tile edges (96 and 97 nodes), K of several
# stages with a one-wide rest (65, 161), odd n_x, the largest K of the 64-bit sums (480 nodes)
MESHES = [(2, 1, 4), (4, 2, 8), (8, 4, 6), (12, 12, 8), (15, 6, 7), (16, 8, 8), (20, 16, 10), (40, 3, 12)]


def _factors(wl, bcset):
    m = wl.mesh
    Kx, Mx = native.operators_1d(m.xb, m.order, True)
    Ky, My = native.operators_1d(m.yb, m.order, False)
    d = np.zeros(len(My), dtype=np.uint8)
    if bcset == native.PF_BCSET_P:
        d[-1] = 1
    Sx, Lx = native.fdm_1d(Kx, Mx)
    Sy, Ly = native.fdm_1d(Ky, My, d)
    Lx[np.abs(Lx) < 1e-11] = 0.0
    Ly[np.abs(Ly) < 1e-11] = 0.0
    return Sx, Lx, Sy, Ly, Mx, My


def _extended(f, factors, shift):
    Sx, Lx, Sy, Ly, Mx, My = (a.astype(np.longdouble) for a in factors)
    b = (Mx[None, :] * My[:, None]).astype(np.float64).astype(np.longdouble)   # the products the solve forms in FP64
    out = []
    for pl in f:
        t = Sy.T @ ((b.astype(np.float64) * pl).astype(np.longdouble)) @ Sx
        out.append(Sy @ (t / (Ly[:, None] + Lx[None, :] + np.longdouble(shift))) @ Sx.T)
    return np.array(out)


@pytest.mark.parametrize("spread", [0, 60])
@pytest.mark.parametrize("mesh", MESHES)
def test_digit_products_are_as_exact_as_fma_chains(mesh, spread):
    """Right-hand sides of equal size and, row by row, of sizes over 60 decades.  The FMA chains' error
    grows with the length of the sums, the digit products' does not (their dropped digits lie 2^-56
    below a product of row maxima), so it may not exceed the chains' by more than the last roundings of
    four products and the reciprocal (1.5 times plus 2e-16)."""
    ex, ey, K = mesh
    wl = workloads.small3d(ex=ex, ey=ey, order=K, nz=4)
    bcset, mode, lam = native.PF_BCSET_P, 1, 2.5
    fac = _factors(wl, bcset)
    ny, nx = len(fac[5]), len(fac[4])
    rng = np.random.default_rng(ex * 100 + K + spread)
    f = rng.standard_normal((2, ny, nx)) * 10.0 ** (spread * (rng.random((2, ny, 1)) - 0.5))
    ref = _extended(f, fac, lam + (2 * np.pi * mode / wl.mesh.lz) ** 2)
    g = native.from_workload(wl, precision=native.PF_FP64)
    err = []
    for gemm in (None, native.PF_GEMM_SIMT32):
        if gemm is not None:
            g.set_variant(gemm, fuse_y=False)
        x = g.solve_helmholtz(bcset, mode, lam, f).reshape(2, ny, nx)
        err.append(float(np.linalg.norm((x - ref).astype(np.float64)) / np.linalg.norm(ref.astype(np.float64))))
    g.close()
    assert err[0] <= 1.5 * err[1] + 2e-16, err
    assert err[0] <= 1e-13


def test_a_non_finite_plane_leaves_the_other_alone():
    wl = workloads.small3d(ex=8, ey=4, order=6, nz=4)
    g = native.from_workload(wl, precision=native.PF_FP64)
    f = np.random.default_rng(3).standard_normal((2, g.ny, g.nx))
    a = g.solve_helmholtz(native.PF_BCSET_U, 1, 1.0, f).reshape(f.shape)
    f[1, 3, 5] = np.nan
    b = g.solve_helmholtz(native.PF_BCSET_U, 1, 1.0, f).reshape(f.shape)
    f[1, 3, 5] = np.inf
    c = g.solve_helmholtz(native.PF_BCSET_U, 1, 1.0, f).reshape(f.shape)
    g.close()
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[0], c[0])
    assert not np.isfinite(b[1]).all() and not np.isfinite(c[1]).all()


@pytest.mark.parametrize("mesh,planes", [((4, 2, 4), 1), ((4, 2, 8), 5), ((8, 4, 6), 1), ((12, 8, 12), 3), ((40, 2, 12), 2)])
def test_static_solve_with_digits(mesh, planes):
    """The allocation-free solve splits the caller's eigenbases in each call: 16 x 9 nodes (FMA kernels),
    32 x 17 and up (digits, also where a row needs padding and K = 480), against extended precision."""
    torch = pytest.importorskip("torch")
    ex, ey, K = mesh
    wl = workloads.small3d(ex=ex, ey=ey, order=K, nz=4)
    fac = _factors(wl, native.PF_BCSET_P)
    Sx, Lx, Sy, Ly, Mx, My = fac
    ny, nx = len(My), len(Mx)
    f = np.random.default_rng(ex + planes).standard_normal((planes, ny, nx))
    t = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")  # noqa: E731
    tables = [t(Sx), t(Sx.T), t(Lx), t(Sy), t(Sy.T), t(Ly)]
    shift, rhs = t(np.full(planes, 3.5)), t((Mx[None, :] * My[:, None]) * f)
    out = torch.empty_like(rhs)
    native.fdm_solve_static(nx, ny, planes, *(x.data_ptr() for x in tables), shift.data_ptr(), rhs.data_ptr(),
                            out.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    ref = _extended(f, fac, 3.5).astype(np.float64)
    assert np.linalg.norm(out.cpu().numpy() - ref) <= 1e-13 * np.linalg.norm(ref)
