"""lb_init and lb_moments of the FP32 and 16-bit lattices at the edges of
their kernels: odd and even widths (one or two columns per thread), ghost
images in x and y, fields and outputs whose addresses do not allow the wide
loads and stores, host arrays in page-locked memory.

Tolerances.  An initial population is the FP64 equilibrium rounded to FP32
once, the arithmetic before it good to about 2^-46: 0.51 units in the last
place.  Density and velocity sum nine FP32 populations and the force (itself
some 30 rounded operations on values below 1): 40 roundings of 2^-24."""
import numpy as np
import pytest

from gpu_util import dev16_solver, oracle_for, solver_for

pytestmark = pytest.mark.gpu

from paper_1307_6703_gb300 import LB_BF16DEV, LB_DTYPE_F32, LB_DTYPE_F64, LB_FP16DEV, LB_FP32, lb_moments  # noqa: E402
from paper_1307_6703_gb300.workloads import C2  # noqa: E402

CX, CY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
W9 = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


def _feq(n, u, v, T):
    uu = u * u + v * v
    out = []
    for i in range(9):
        cu, cc = CX[i] * u + CY[i] * v, CX[i] ** 2 + CY[i] ** 2
        out.append(W9[i] * n * (1 + 3 * cu + 4.5 * (cu * cu - uu / 3) + 4.5 * (T - 1 / 3) * (cc - 2 / 3)))
    return np.stack(out)


def _w(nx, ny, walls):
    u = 0.03 if walls else 0.0
    return C2(0.05).with_(nx=nx, ny=ny, walls=walls, A0=3e-4, lam=32.0, u_bot=-u, u_top=u)


def _fields(nx, ny):
    r = np.random.default_rng(nx + 1000 * ny)
    return 1 + 0.4 * r.uniform(-1, 1, (ny, nx)), 0.1 * r.uniform(-1, 1, (ny, nx)), 0.1 * r.uniform(-1, 1, (ny, nx))


@pytest.mark.parametrize("nx,ny,walls", [(5, 3, True), (8, 8, False), (61, 20, True), (62, 20, False), (64, 9, True),
                                         (300, 33, False)])
@pytest.mark.parametrize("given", ["n", "n,u", "n,u,v"])
def test_initial_populations_are_the_rounded_equilibrium(nx, ny, walls, given):
    w = _w(nx, ny, walls)
    f = dict(zip("nuv", _fields(nx, ny)))
    args = [f[k] if k in given.split(",") else None for k in "nuv"]
    zero = np.zeros((ny, nx))
    ref = _feq(args[0], *[zero if a is None else a for a in args[1:]], w.T)
    s = solver_for(w, LB_FP32).init_fields(*args)
    got = s.get_state()
    assert np.all(np.abs(got.astype(np.float64) - ref) <= 0.51 * np.spacing(np.abs(ref).astype(np.float32)))
    # device fields at an odd address (8 modulo 16) give the same bits
    import torch
    dev = [None if a is None else torch.empty(nx * ny + 1, dtype=torch.float64, device="cuda")[1:].view(ny, nx) for a in args]
    for d, a in zip(dev, args):
        if d is not None:
            d.copy_(torch.from_numpy(a))
    assert np.array_equal(solver_for(w, LB_FP32).init_fields(*dev).get_state(), got)
    # the ghost band is right: a step from it equals a step from a restored state
    t = solver_for(w, LB_FP32)
    t.set_state(got)
    assert np.array_equal(t.step(1).get_state(), s.step(1).get_state())


@pytest.mark.parametrize("prec", [LB_FP32, LB_BF16DEV, LB_FP16DEV], ids=["fp32", "bf16dev", "fp16dev"])
@pytest.mark.parametrize("nx,ny,walls", [(8, 8, False), (56, 11, True), (120, 40, False), (304, 65, True)])
def test_moments_and_their_destinations(prec, nx, ny, walls):
    import torch
    w = _w(nx, ny, walls)
    n0 = _fields(nx, ny)[0]
    s = (solver_for(w, prec) if prec == LB_FP32 else dev16_solver(w, prec, 1.0)).init_fields(n0)
    dev = torch.empty((3, ny, nx), dtype=torch.float32, device="cuda")
    lb_moments(s.h, dev[0], dev[1], dev[2], LB_DTYPE_F32, 1)
    got = dev.cpu().numpy()
    if prec == LB_FP32:
        ref = oracle_for(w).init_fields(n0).moments()
        for g, r in zip(got, ref):
            assert np.abs(g - r).max() <= 40 * 2.0 ** -24 * np.abs(ref[0]).max()
    # FP64 outputs are the same values; odd addresses, host and page-locked arrays, single outputs
    d64 = torch.empty((3, ny, nx), dtype=torch.float64, device="cuda")
    lb_moments(s.h, d64[0], d64[1], d64[2], LB_DTYPE_F64, 1)
    assert np.array_equal(d64.cpu().numpy(), got.astype(np.float64))
    odd = torch.full((3 * nx * ny + 1,), -7.0, dtype=torch.float32, device="cuda")
    o = odd[1:].view(3, ny, nx)
    lb_moments(s.h, o[0], o[1], o[2], LB_DTYPE_F32, 1)
    assert np.array_equal(o.cpu().numpy(), got) and odd[0].item() == -7.0
    pin = torch.empty((3, ny, nx), dtype=torch.float32).pin_memory()
    lb_moments(s.h, pin[0], pin[1], pin[2], LB_DTYPE_F32, 0)
    assert np.array_equal(pin.numpy(), got)
    assert all(np.array_equal(a, b) for a, b in zip(s.moments(np.float32), got))
    only = torch.empty((ny, nx), dtype=torch.float32, device="cuda")
    lb_moments(s.h, None, only, None, LB_DTYPE_F32, 1)
    assert np.array_equal(only.cpu().numpy(), got[1])
