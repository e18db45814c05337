"""Rounding of lb_moments in FP32 and 16-bit storage.  The formulas written down
plainly in numpy, every operation in FP32, are one way of reading a state; the
kernel must not be further from the same formulas in FP64 than that (root mean
square over the lattice: tens of thousands of independent roundings, so equal
forms agree within a few per cent; 5 % allowed)."""
import numpy as np
import pytest

from gpu_util import decode_state, dev16_solver, solver_for

pytestmark = pytest.mark.gpu

from paper_1307_6703_gb300 import LB_BF16DEV, LB_FP16DEV, LB_FP32  # noqa: E402
from paper_1307_6703_gb300.workloads import C2  # noqa: E402


def _moments(w, f, t):
    """Density and velocity of populations f (periodic), every operation in t."""
    cx, cy = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
    f = [np.roll(f[i].astype(t), (cy[i], cx[i]), (0, 1)) for i in range(9)]
    at = lambda a, dx, dy: np.roll(a, (-dy, -dx), (0, 1))  # noqa: E731
    a, b, T, k, N, Q = (t(v) for v in (w.a, w.b, w.T, w.kappa, w.N, w.Q))
    M, R, half = t((1 - 2 * w.N) / 4), t((1 - w.Q) / 2), t(0.5)

    def grad(p):
        p = [at(p, cx[i], cy[i]) for i in range(9)]
        return (N * (p[1] - p[3]) + M * ((p[5] - p[6]) + (p[8] - p[7])), N * (p[2] - p[4]) + M * ((p[5] - p[8]) + (p[6] - p[7])))
    n = f[0]
    for i in range(1, 9):
        n = n + f[i]
    p = [at(n, cx[i], cy[i]) for i in range(9)]
    L = (Q * (((p[1] + p[2]) + p[3]) + p[4]) + R * (((p[5] + p[6]) + p[7]) + p[8])) - t(4) * (Q + R) * n
    P = n * T - ((n * T) / (t(1) - b * n) - a * n * n)
    (Px, Py), (Lx, Ly) = grad(P), grad(L)
    fx = (w.A0 * np.sin(2 * np.pi * np.arange(w.nx) / w.lam)).astype(t)[None, :]
    Fx, Fy = (Px + k * n * Lx) + fx, Py + k * n * Ly
    sx = ((((f[1] - f[3]) + f[5]) - f[6]) - f[7]) + f[8]
    sy = ((((f[2] - f[4]) + f[5]) + f[6]) - f[7]) - f[8]
    return n, (sx + half * Fx) / n, (sy + half * Fy) / n


@pytest.mark.parametrize("prec,nx,ny", [(LB_FP32, 256, 128), (LB_FP32, 253, 130), (LB_BF16DEV, 256, 128), (LB_FP16DEV, 264, 130)])
@pytest.mark.parametrize("start", ["rest", "moving"])
def test_moments_round_as_little_as_their_formulas(prec, nx, ny, start):
    w = C2(0.05).with_(nx=nx, ny=ny, walls=False, A0=3e-4, lam=32.0, u_bot=0.0, u_top=0.0)
    rng = np.random.default_rng(nx + ny)
    y, x = np.mgrid[0:ny, 0:nx]
    n0 = 1.0 + 0.3 * np.sin(2 * np.pi * y / ny + 0.3) * np.cos(2 * np.pi * x / nx) + 0.01 * rng.uniform(-1, 1, (ny, nx))
    u0 = (0.05 * np.sin(2 * np.pi * y / ny + 1.0),) * (2 if start == "moving" else 0)
    s = (solver_for(w, prec) if prec == LB_FP32 else dev16_solver(w, prec, 1.0)).init_fields(n0, *u0).step(3)
    f = s.get_state()
    if prec != LB_FP32:
        f = decode_state(f[0], f[1], "bf16" if prec == LB_BF16DEV else "fp16", 1.0)
    for g, r, e in zip(s.moments(), _moments(w, f, np.float32), _moments(w, f, np.float64)):
        assert np.sqrt(np.mean((g - e) ** 2)) <= 1.05 * np.sqrt(np.mean((r.astype(np.float64) - e) ** 2))
    s.close()
