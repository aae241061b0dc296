"""Fields read into pinned memory (one kernel stores them there) against the same fields read into pageable memory."""
import numpy as np
import pytest

import workloads
from paper_2305_09020_gb300 import native

pytestmark = pytest.mark.gpu

F = native
MASKS = [F.PF_FIELD_V, F.PF_FIELD_E | F.PF_FIELD_P, F.PF_FIELD_V | F.PF_FIELD_PHI | F.PF_FIELD_PSI | F.PF_FIELD_U,
         F.PF_FIELD_V | F.PF_FIELD_E | F.PF_FIELD_PHI | F.PF_FIELD_P | F.PF_FIELD_U,
         F.PF_FIELD_OLD | F.PF_FIELD_PHI | F.PF_FIELD_U]


@pytest.mark.parametrize("mask", MASKS)
@pytest.mark.parametrize("nz", [1, 6])
@pytest.mark.parametrize("precision", [native.PF_FP64, native.PF_MIXED])
def test_pinned_buffer_gets_the_same_bits(precision, nz, mask):
    """Every selection, with fields that a 2D run does not hold (zeros) and with psi (formed on the host);
    the buffer starts inside its allocation and ends with it, and what lies before it stays."""
    import torch
    wl = workloads.small3d(ex=3, ey=2, order=5, nz=6) if nz > 1 else workloads.small2d(ex=3, ey=2, order=5)
    g = native.from_workload(wl, precision=precision)
    g.step(2)
    want = np.concatenate([v.ravel() for v in g.get(mask).values()])
    pin = torch.full((want.size + 3,), -7.0, dtype=torch.float64, pin_memory=True)
    assert pin.is_pinned()
    g.get_into(mask, pin.numpy()[3:])
    g.close()
    assert np.array_equal(pin.numpy()[3:], want)
    assert (pin.numpy()[:3] == -7.0).all()
