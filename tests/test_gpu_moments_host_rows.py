"""Moments of odd-width lattices in page-locked host arrays are the bits of those in
device arrays: widths around one and two rows of 32 columns, and each array alone."""
import numpy as np
import pytest

from gpu_util import solver_for

pytestmark = pytest.mark.gpu

from paper_1307_6703_gb300 import LB_DTYPE_F32, LB_DTYPE_F64, LB_FP32, lb_moments  # noqa: E402
from paper_1307_6703_gb300.workloads import C2  # noqa: E402


@pytest.mark.parametrize("nx,ny", [(9, 8), (31, 9), (33, 12), (34, 8), (63, 11), (65, 10), (66, 9), (67, 8), (99, 33), (1021, 40)])
@pytest.mark.parametrize("dtype", [LB_DTYPE_F32, LB_DTYPE_F64])
def test_host_arrays_hold_the_same_bits(nx, ny, dtype):
    import torch
    w = C2(0.05).with_(nx=nx, ny=ny, A0=3e-4, lam=32.0)
    r = np.random.default_rng(nx)
    s = solver_for(w, LB_FP32).init_fields(1 + 0.3 * r.uniform(-1, 1, (ny, nx))).step(2)
    t = torch.float32 if dtype == LB_DTYPE_F32 else torch.float64
    d = torch.full((3, ny, nx), -7.0, dtype=t, device="cuda")
    h = torch.full((3, ny, nx), -7.0, dtype=t).pin_memory()
    lb_moments(s.h, d[0], d[1], d[2], dtype, 1)
    lb_moments(s.h, h[0], h[1], h[2], dtype, 0)
    torch.cuda.synchronize()
    assert torch.equal(d.cpu(), h)
    for k in range(3):
        one = torch.full((ny + 2, nx), -7.0, dtype=t).pin_memory()   # (rows before and after stay as they are)
        lb_moments(s.h, *[one[1:-1] if i == k else None for i in range(3)], dtype, 0)
        assert torch.equal(one[1:-1], h[k]) and bool((one[[0, -1]] == -7.0).all())
    s.close()
