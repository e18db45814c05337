"""Initial state, steps and moments queued without synchronisation: each kernel
is scheduled before the one ahead of it has finished and waits for it, so
passes of different seeds, one behind the other on one state, give the bits of
each pass on its own.  Sizes: one tile, a few, and more tiles than the device
holds warps (blocks of the next kernel then wait behind the last ones of this);
steps 1 (single launches), 2 (multi-step) and both."""
import pytest

from gpu_util import dev16_solver, solver_for

pytestmark = pytest.mark.gpu

from paper_1307_6703_gb300 import LB_BF16DEV, LB_DTYPE_F32, LB_FP32, lb_moments  # noqa: E402
from paper_1307_6703_gb300.workloads import C2  # noqa: E402


@pytest.mark.parametrize("prec", [LB_FP32, LB_BF16DEV])
@pytest.mark.parametrize("nx,ny,walls", [(16, 8, True), (200, 40, False), (203, 37, True), (2048, 600, True)])
def test_queued_passes_give_the_bits_of_each_alone(prec, nx, ny, walls):
    import torch
    if prec == LB_BF16DEV and nx % 8:
        pytest.skip("16-bit storage takes multiples of 8 columns")
    u = 0.03 if walls else 0.0
    w = C2(0.05).with_(nx=nx, ny=ny, walls=walls, A0=3e-4, lam=32.0, u_bot=-u, u_top=u)
    s = dev16_solver(w, prec, 1.0) if prec == LB_BF16DEV else solver_for(w, prec)

    def one(seed, steps, m):
        s.init_noise(seed=seed, rho_mean=1.0, amp=0.003)
        for k in steps:
            s.step(k)
        lb_moments(s.h, m[0], m[1], m[2], LB_DTYPE_F32, 1)

    passes = [(1, ()), (2, (1,)), (3, (2,)), (4, (1, 2, 1)), (5, (1, 1, 1)), (6, ())] * 3
    alone, queued = [[torch.empty((3, ny, nx), dtype=torch.float32, device="cuda") for _ in passes] for _ in range(2)]
    for (seed, steps), m in zip(passes, alone):
        one(seed, steps, m)
        torch.cuda.synchronize()
    for (seed, steps), m in zip(passes, queued):
        one(seed, steps, m)
    torch.cuda.synchronize()
    for a, b in zip(alone, queued):
        assert torch.isfinite(a).all() and torch.equal(a, b)
