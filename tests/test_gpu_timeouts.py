"""A bounded device wait that gives up (the test hook's, on a barrier that nothing arrives at) is reported by every
call that reads results: FP64 runs on the digit transforms, and ensembles in both precisions."""
import numpy as np
import pytest

import workloads
from paper_2305_09020_gb300 import native

pytestmark = pytest.mark.gpu

WAIT = 20_000_000   # 20 ms


def _times_out(call):
    with pytest.raises(native.PfError) as ei:
        call()
    assert ei.value.code == native.PF_ETIMEOUT


def test_fp64_run():
    wl = workloads.small2d(ex=8, ey=4, order=6)      # 48 x 25 nodes
    h = native.from_workload(wl, precision=native.PF_FP64)
    f = np.random.default_rng(3).standard_normal((h.ny, h.nx))
    good = h.solve_helmholtz(native.PF_BCSET_NN, 0, 1.5, f)
    h.debug_tc_stall(WAIT)
    _times_out(lambda: h.solve_helmholtz(native.PF_BCSET_NN, 0, 1.5, f))
    assert np.array_equal(h.solve_helmholtz(native.PF_BCSET_NN, 0, 1.5, f), good)
    h.step(2)
    h.debug_tc_stall(WAIT)
    h.step(1)
    _times_out(lambda: h.get(native.PF_FIELD_PHI))
    _times_out(h.diagnostics)
    _times_out(h.sync)                               # clears it
    h.get(native.PF_FIELD_PHI)
    h.close()


def test_fp64_run_without_tensor_cores_refuses_the_hook():
    h = native.from_workload(workloads.small2d(ex=4, ey=2, order=4), precision=native.PF_FP64)
    with pytest.raises(native.PfError) as ei:
        h.debug_tc_stall(WAIT)
    assert ei.value.code == native.PF_EINVAL
    h.close()


@pytest.mark.parametrize("precision", [native.PF_FP64, native.PF_MIXED])
@pytest.mark.parametrize("call", ["get", "umax", "march", "autotune"])
def test_ensemble(precision, call):
    runs = [workloads.small2d(ex=ex, ey=ex // 2, order=6) for ex in (8, 6, 8)]
    b = native.Batch(runs, precision=precision)
    b.step(2)
    b.umax()
    b.debug_tc_stall(WAIT)
    if call == "march":
        _times_out(lambda: b.run_to_equilibrium(0.0, 4, 2))
    elif call == "autotune":
        _times_out(lambda: b.autotune(1))
    else:
        b.step(1)
        _times_out((lambda: b.get(0, native.PF_FIELD_PHI)) if call == "get" else b.umax)
    _times_out(lambda: b.step(1))                    # known by now
    b.close()
