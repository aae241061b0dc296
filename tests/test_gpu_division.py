"""The eigenvalue division of the tensor-core transforms on both sides of the range of its branch-free form."""
import numpy as np
import pytest

import workloads
from paper_2305_09020_gb300 import native

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mesh", [(6, 5, 6), (16, 8, 8)])
@pytest.mark.parametrize("lam", [1e13, 1e16, 1e20])
def test_large_shifts(mesh, lam):
    """(K + lam M) x = M f between Neumann walls: x = f / lam up to the largest eigenvalue of M^-1 K (below
    3e5 on these meshes) over lam, far less than the FP32 bar of a solve (2e-6)."""
    ex, ey, K = mesh
    wl = workloads.small3d(ex=ex, ey=ey, order=K, nz=4)
    g = native.from_workload(wl, precision=native.PF_MIXED)
    g.set_variant(native.PF_GEMM_TC, fuse_y=False)
    f = np.random.default_rng(K).standard_normal((2, wl.mesh.ex * K * (wl.mesh.ey * K + 1)))
    x = g.solve_helmholtz(native.PF_BCSET_NN, 1, lam, f).reshape(f.shape)
    g.close()
    assert np.linalg.norm(x * lam - f) <= 2e-6 * np.linalg.norm(f)
