"""Infinities and NaN in the caller's eigenbases of the allocation-free solve."""
import numpy as np
import pytest

import workloads
from paper_2305_09020_gb300 import native

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("mesh", [(4, 2, 4), (8, 4, 6)])   # 16 x 9 nodes: FMA kernels; 48 x 25: digits
@pytest.mark.parametrize("which", [0, 1, 3, 4])            # Sx, SxT, Sy, SyT
def test_static_solve_reports_a_broken_eigenbasis(mesh, which, bad):
    """One bad entry of one eigenbasis, opposite right-hand sides that are zero but for a few nodes: every sum
    that meets the entry is NaN or infinite (0 times it is NaN), so with Sx or Sy no result is finite, with a
    transpose the column or row it belongs to is not and the others are those of the sound basis (to the rounding
    of the four products, whose scaling may depend on the entry)."""
    torch = pytest.importorskip("torch")
    wl = workloads.small3d(ex=mesh[0], ey=mesh[1], order=mesh[2], nz=4)
    m = wl.mesh
    Kx, Mx = native.operators_1d(m.xb, m.order, True)
    Ky, My = native.operators_1d(m.yb, m.order, False)
    Sx, Lx = native.fdm_1d(Kx, Mx)
    Sy, Ly = native.fdm_1d(Ky, My)
    nx, ny = len(Mx), len(My)
    f = np.zeros((2, ny, nx))
    f[:, ny // 2, nx // 3] = [1.0, -1e-200]

    def solve(tables):
        t = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")  # noqa: E731
        dev = [t(a) for a in tables]
        shift, rhs = t(np.full(2, 3.5)), t(f)
        out = torch.zeros_like(rhs)
        native.fdm_solve_static(nx, ny, 2, *(x.data_ptr() for x in dev), shift.data_ptr(), rhs.data_ptr(),
                                out.data_ptr(), torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        return out.cpu().numpy()

    tables = [Sx, Sx.T, np.abs(Lx), Sy, Sy.T, np.abs(Ly)]
    good = solve(tables)
    assert np.isfinite(good).all()
    i, j = 2, 5                                  # row k = 2, column n = 5 of the table
    tables[which] = tables[which].copy()
    tables[which][i, j] = bad
    x = solve(tables)
    if which in (0, 3):
        assert not np.isfinite(x).any()
    elif which == 1:                             # out[.., n] = sum_k W[.., k] SxT[k, n]
        assert not np.isfinite(x[:, :, j]).any()
        assert np.abs(np.delete(x - good, j, axis=2)).max() <= 1e-13 * np.abs(good).max()
    else:                                        # W1[n, ..] = sum_k W2[.., k] SyT[k, n]
        assert not np.isfinite(x[:, j, :]).any()
        assert np.abs(np.delete(x - good, j, axis=1)).max() <= 1e-13 * np.abs(good).max()
