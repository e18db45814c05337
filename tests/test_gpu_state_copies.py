"""States of padded handles set from and read into host memory, in one and in
several pieces: what was set is read back bit for bit, and the density of the
state on the device is that of the array that was set, streamed on the host
(periodic; FP32: nine roundings of a sum of nine populations; 16-bit storage:
the decoded deviations, the same)."""
import numpy as np
import pytest

from gpu_util import decode_state, dev16_solver, solver_for

pytestmark = pytest.mark.gpu

from paper_1307_6703_gb300 import LB_BF16DEV, LB_FP16DEV, LB_FP32  # noqa: E402
from paper_1307_6703_gb300.workloads import C2  # noqa: E402

CX, CY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)


@pytest.mark.parametrize("prec,nx,ny", [(LB_FP32, 9, 8), (LB_FP32, 57, 33), (LB_FP32, 1021, 2100), (LB_FP32, 1024, 2100),
                                        (LB_FP32, 99999, 11), (LB_BF16DEV, 8, 8), (LB_BF16DEV, 1024, 4200),
                                        (LB_FP16DEV, 136, 57)])
def test_states_set_and_read(prec, nx, ny):
    w = C2(0.05).with_(nx=nx, ny=ny, walls=False, u_bot=0.0, u_top=0.0, lam=32.0)
    rng = np.random.default_rng(nx + ny)
    if prec == LB_FP32:
        s = solver_for(w, prec)
        f = rng.uniform(0.05, 0.15, (9, ny, nx)).astype(np.float32)
        s.set_state(f)
        assert np.array_equal(s.get_state(), f)
    else:
        s = dev16_solver(w, prec, 1.0)
        f0 = rng.uniform(0.3, 0.5, (ny, nx)).astype(np.float32)
        v = rng.uniform(-0.02, 0.02, (8, ny, nx)).astype(np.float32)
        d = (v.view(np.uint32) >> 16).astype(np.uint16) if prec == LB_BF16DEV else v.astype(np.float16).view(np.uint16)
        s.set_state((f0, d))
        g0, g = s.get_state()
        assert np.array_equal(g0, f0) and np.array_equal(g, d)
        f = decode_state(f0, d, "bf16" if prec == LB_BF16DEV else "fp16", 1.0)
    n = sum(np.roll(f[i].astype(np.float64), (CY[i], CX[i]), (0, 1)) for i in range(9))
    assert np.abs(s.moments()[0] - n).max() <= 9 * 2.0 ** -24 * n.max()
    s.close()
