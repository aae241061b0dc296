"""The digit transforms as a variant by its own code: pinned, left and taken up again, and named by the autotuner."""
import numpy as np
import pytest

import workloads
from paper_2305_09020_gb300 import native

pytestmark = pytest.mark.gpu


def _solve(h):
    f = np.random.default_rng(7).standard_normal((h.ny, h.nx))
    return h.solve_helmholtz(native.PF_BCSET_U, 0, 1.0, f)


def test_a_run_returns_to_its_default():
    h = native.from_workload(workloads.small2d(ex=8, ey=4, order=6), precision=native.PF_FP64)
    default = _solve(h)
    h.set_variant(native.PF_GEMM_SIMT32, fuse_y=False)
    assert not np.array_equal(_solve(h), default)        # other roundings: another kernel ran
    h.set_variant(native.PF_GEMM_DIGITS)
    assert np.array_equal(_solve(h), default)
    h.close()


@pytest.mark.parametrize("mesh", [(8, 4, 6), (15, 6, 7)])
def test_an_autotuned_choice_can_be_reproduced(mesh):
    """The choice, pinned on another run, gives the bits of the run that was tuned."""
    wl = workloads.small2d(ex=mesh[0], ey=mesh[1], order=mesh[2])
    a = native.from_workload(wl, precision=native.PF_FP64)
    choice, ms = a.autotune(steps=3)
    gemm, tile, fused = choice % 1000, (choice // 1000) % 100, choice // 100000
    b = native.from_workload(wl, precision=native.PF_FP64)
    b.set_variant(gemm, fuse_y=bool(fused), tile=tile)
    assert ms > 0 and np.array_equal(_solve(a), _solve(b)), choice
    a.close()
    b.close()


def test_runs_without_digit_transforms_refuse_the_code():
    small = workloads.small2d(ex=4, ey=2, order=4)
    for h in (native.from_workload(small, precision=native.PF_FP64),
              native.from_workload(workloads.small2d(ex=8, ey=4, order=6), precision=native.PF_MIXED)):
        with pytest.raises(native.PfError) as ei:
            h.set_variant(native.PF_GEMM_DIGITS)
        assert ei.value.code == native.PF_EINVAL
        h.close()


def test_ensemble_pins_digits_where_every_group_has_them():
    wide, small = [workloads.small2d(ex=e, ey=2, order=6) for e in (8, 6)], workloads.small2d(ex=4, ey=2, order=4)
    b = native.Batch(wide, precision=native.PF_FP64)
    b.set_variant(native.PF_GEMM_SIMT64)
    b.set_variant(native.PF_GEMM_DIGITS)
    b.step(2)
    assert np.all(b.autotune(steps=1) > 0)
    b.close()
    b = native.Batch([*wide, small], precision=native.PF_FP64)
    with pytest.raises(native.PfError) as ei:
        b.set_variant(native.PF_GEMM_DIGITS)
    assert ei.value.code == native.PF_EINVAL
    b.close()
