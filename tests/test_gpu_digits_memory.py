"""An FP64 run whose device memory holds the run but not the digits of its transforms."""
import numpy as np
import pytest

import workloads
from gpu_util import ALL
from paper_2305_09020_gb300 import native

pytestmark = pytest.mark.gpu


def test_a_run_that_fits_without_the_digits_is_created():
    torch = pytest.importorskip("torch")
    wl = workloads.small3d(ex=24, ey=12, order=8, nz=64)
    kpad = lambda k: (k + 31) // 32 * 32  # noqa: E731
    nx, ny, nz = 192, 97, 64
    digits = 16 * 3 * nz * max(ny * kpad(nx), nx * kpad(ny)) + 16 * 5 * (nz // 2 + 1) * nx * ny   # 110 MB
    warm = native.from_workload(wl, precision=native.PF_FP64)      # every kernel of both forms is loaded
    warm.step(3)
    ref = warm.get(ALL)
    warm.set_variant(native.PF_GEMM_SIMT32)
    warm.step(1)
    warm.close()
    free0, _ = torch.cuda.mem_get_info()
    h = native.from_workload(wl, precision=native.PF_FP64)
    used = free0 - torch.cuda.mem_get_info()[0]
    h.close()
    assert used > 2 * digits
    free0, _ = torch.cuda.mem_get_info()
    filler = torch.empty(free0 - used + digits // 2, dtype=torch.uint8, device="cuda")
    try:
        h = native.from_workload(wl, precision=native.PF_FP64)
        with pytest.raises(native.PfError):
            h.set_variant(native.PF_GEMM_DIGITS)                    # it runs on the FMA transforms
        h.step(3)
        got = h.get(ALL)
        h.close()
    finally:
        del filler
        torch.cuda.empty_cache()
    for k in ref:
        assert np.linalg.norm(got[k] - ref[k]) <= 1e-11 * max(np.linalg.norm(ref[k]), 1e-30), k
