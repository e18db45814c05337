"""FP32 lattices whose width is not a multiple of 4: the sweep's last tile is
narrower, ends in half a pair of columns for odd widths, and periodic images
are stored by columns.  Widths around one and two tiles (56 columns) and every
remainder, single and multi-step launches, walls and periodic rows, both forms
of the relaxation, moments to device and host, states set and read back, and
steps captured in a graph, against the FP64 oracle.

Tolerance: a step rounds each population about 25 times (relative 2^-24
each), so five steps stay below 5 * 25 * 6e-8 = 7.5e-6 of the largest
population even if every rounding went the same way; a moment adds nine of
them (nine more roundings of sums of at most nine populations)."""
import numpy as np
import pytest

from gpu_util import oracle_for, rel_err, solver_for

pytestmark = pytest.mark.gpu

from paper_1307_6703_gb300 import LB_FP32, Batch, LBError, lb_get_tiling  # noqa: E402
from paper_1307_6703_gb300.workloads import C2  # noqa: E402

STEPS, TOL = 5, 5 * 25 * 2.0 ** -24


def _w(nx, ny, walls, tau):
    u = 0.04 if walls else 0.0
    return C2(0.05).with_(nx=nx, ny=ny, walls=walls, tau=tau, A0=3e-4, lam=32.0, u_bot=-u, u_top=u)


def _n0(nx, ny):
    rng = np.random.default_rng(nx * 1000 + ny)
    y, x = np.mgrid[0:ny, 0:nx]
    return 1.0 + 0.3 * np.sin(2 * np.pi * y / ny) * np.cos(2 * np.pi * x / nx) + 0.01 * rng.uniform(-1, 1, (ny, nx))


@pytest.mark.parametrize("tau", [1.0, 2.0])
@pytest.mark.parametrize("walls", [True, False], ids=["walls", "periodic"])
@pytest.mark.parametrize("nx,ny", [(9, 8), (10, 9), (11, 31), (53, 10), (57, 11), (58, 8), (59, 12), (111, 13),
                                   (113, 33), (114, 16), (299, 67)])
def test_odd_widths_against_the_oracle(nx, ny, walls, tau):
    w = _w(nx, ny, walls, tau)
    n0 = _n0(nx, ny)
    s = solver_for(w, LB_FP32).init_fields(n0).step(STEPS)
    ref = oracle_for(w).init_fields(n0).step(STEPS)
    f = s.get_state()
    assert rel_err(f, ref.f) <= TOL
    one = solver_for(w, LB_FP32).init_fields(n0)
    for _ in range(STEPS):
        one.step(1)
    assert np.array_equal(one.get_state(), f)  # single steps: the same bits
    back = solver_for(w, LB_FP32)
    back.set_state(f)
    assert np.array_equal(back.step(2).get_state(), one.step(2).get_state())
    ref.step(2)
    for g, r in zip(one.moments(), ref.moments()):
        assert np.abs(g - r).max() <= 2 * (STEPS + 2) / STEPS * 9 * TOL
    mass = one.reduce()[1][0]
    assert abs(mass - ref.f.sum()) <= 2 * TOL * ref.f.sum()
    for h in (s, one, back):
        h.close()


def test_odd_widths_have_no_tiling_and_join_no_batch():
    import torch
    w = _w(57, 20, True, 1.0)
    s = solver_for(w, LB_FP32)
    assert lb_get_tiling(s.h) == (0, 0)
    with pytest.raises(LBError):
        s.monitor(torch.zeros((16, 6), dtype=torch.float64, device="cuda"), 16)
    with pytest.raises(LBError):
        Batch([s.params])
    s.close()


@pytest.mark.parametrize("nx", [57, 58])
def test_odd_widths_step_inside_a_capture(nx):
    import torch
    from paper_1307_6703_gb300 import Solver
    w = _w(nx, 20, False, 1.0)
    n0 = _n0(nx, 20)
    st = torch.cuda.Stream()
    s = Solver(w.nx, w.ny, precision=LB_FP32, walls=w.walls, a=w.a, b=w.b, T=w.T, kappa=w.kappa, tau=w.tau, A0=w.A0,
               lam=w.lam, u_bot=w.u_bot, u_top=w.u_top, N=w.N, Q=w.Q, stream=st.cuda_stream)
    s.init_fields(n0).step(2)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        s.step(4)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    ref = solver_for(w, LB_FP32).init_fields(n0).step(14)
    assert np.array_equal(s.get_state(), ref.get_state())
    s.close()
