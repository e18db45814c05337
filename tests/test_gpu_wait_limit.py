"""A single step in which every copy wait gives up (lb_set_wait_limit 0: the
kernel stops early, within bounds): the sums say so instead of returning those
of the step before, and the context and other handles go on."""
import numpy as np
import pytest

from gpu_util import dev16_solver, solver_for

pytestmark = pytest.mark.gpu

from paper_1307_6703_gb300 import (LB_BF16DEV, LB_ERR_TIMEOUT, LB_FP32, LBError, lb_reduce_async,  # noqa: E402
                                   lb_set_wait_limit)
from paper_1307_6703_gb300.workloads import C2  # noqa: E402


@pytest.mark.parametrize("prec,nx,ny", [(LB_FP32, 64, 32), (LB_FP32, 512, 256), (LB_BF16DEV, 64, 32), (LB_FP32, 57, 20)])
@pytest.mark.parametrize("tau", [1.0, 2.0])
@pytest.mark.parametrize("monitored", [False, True])  # (then the last tile adds the records up)
def test_a_single_step_that_gives_up_is_reported(prec, nx, ny, tau, monitored):
    if monitored and nx % 4:
        pytest.skip("no monitoring of these widths")
    import torch
    w = C2(0.05).with_(nx=nx, ny=ny, tau=tau, lam=32.0)
    make = (lambda: solver_for(w, prec)) if prec == LB_FP32 else (lambda: dev16_solver(w, prec, 1.0))
    s = make().init_noise(1, 1.0, 0.01)
    if monitored:
        ring = torch.zeros((16, 6), dtype=torch.float64).pin_memory()
        s.monitor(ring)
    s.step(1)
    assert s.reduce()[0] == 0
    lb_set_wait_limit(s.h, 0)
    s.step(1)
    out = torch.zeros(5, dtype=torch.float64).pin_memory()
    lb_reduce_async(s.h, out)
    torch.cuda.synchronize()
    assert float(out[4]) == 1.0
    lb_set_wait_limit(s.h, 1 << 22)
    for _ in range(3):  # and for the rest of the handle's life
        with pytest.raises(LBError) as e:
            s.reduce()
        assert e.value.code == LB_ERR_TIMEOUT
        s.step(1)
    s.close()
    a, b = make().init_noise(1, 1.0, 0.01).step(4), make().init_noise(1, 1.0, 0.01).step(4)
    assert a.reduce()[0] == 0
    fa, fb = a.get_state(), b.get_state()
    assert all(np.array_equal(x, y) for x, y in zip(fa, fb))
    a.close()
    b.close()
